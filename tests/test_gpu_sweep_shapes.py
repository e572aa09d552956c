"""Sweeps at the edges of every kernel shape against the CPU oracle, bit for bit.

A row is decided in passes of 16, 32, 64 or 128 sites (Ising up to 16 x 16: site by
site), so the sides here are the smallest and largest of each shape, their neighbours,
and sides that leave one to three sites in a row's last lane.  The thresholds are those
of weights with noise of 0.3 per bin, which makes many passes need repairs; every chain
runs on both sides with the same table, so nothing but equality is allowed.
"""
import numpy as np
import pytest

import workloads
from oracle import MucaOracle, reweight, weights

pytestmark = pytest.mark.gpu

ISING, POTTS = 0, 1
SIDES = [(ISING, L) for L in (4, 6, 10, 12, 14, 16, 18, 20, 30, 32, 34, 62, 66, 126, 128, 130, 132, 162, 226, 258)] \
    + [(POTTS, L) for L in (3, 4, 7, 16, 17, 18, 19, 31, 33, 63, 64, 65, 127, 129, 130, 131, 255)]


@pytest.fixture(scope="module")
def muca():
    import paper_1212_3975_gb300 as m
    from paper_1212_3975_gb300 import build
    build.build()
    return m


def noisy_thresholds(model, L):
    lnw = workloads.canonical_lnw(model, L, 0.3 if model == ISING else 1.2) + workloads.random_lnw(model, L, L, 0.3)
    return weights.thresholds(model, L, np.where(weights.accessible(model, L), lnw, 0.0))


@pytest.mark.parametrize("model,L", SIDES)
@pytest.mark.parametrize("staging", [0, 2])
def test_every_shape_bit_exact(muca, model, L, staging):
    """Two iterations, thermalisation and production with lattices in shared (0) and
    global (2) memory; a ragged number of chains, so that warps hold padding chains."""
    p = 3 if L > 128 else 11
    sweeps = 1 if L > 128 else max(2, 2000 // (L * L))
    q = 2 if model == ISING else 8
    thr = noisy_thresholds(model, L)
    with muca.Muca(model, L, q, p, 77, staging=staging) as g:
        g.set_thresholds(thr)
        H1 = g.iterate(sweeps)
        H2 = g.iterate(1)
        g.thermalize(sweeps)
        E, M = g.produce(2)
        n, s1, s2 = g.get_samples()
        spins = g.get_spins()
        E_end, M_end = g.get_energies()
    o = MucaOracle(model, L, q, p, 77)
    assert np.array_equal(H1, o.iterate(sweeps, thr=thr))
    assert np.array_equal(H2, o.iterate(1, thr=thr))
    o.thermalize(sweeps, thr=thr)
    e, m = o.produce(2, thr=thr)
    assert np.array_equal(E, e) and np.array_equal(M, m)
    for x, y in zip((n, s1, s2), reweight.bin_series(model, L, e, m)):
        assert np.array_equal(x, y)
    assert np.array_equal(spins, o.spins)
    assert np.array_equal(E_end, o.E) and np.array_equal(M_end, o.M)


@pytest.mark.parametrize("model,L,groups", [(ISING, 8, 700), (ISING, 32, 700), (ISING, 64, 450), (POTTS, 8, 700),
                                            (POTTS, 32, 650)])
def test_many_chains_bit_exact(muca, model, L, groups):
    """Several blocks of several groups (more deciding than drawing warps) and a ragged
    last block; sampled chains are replayed by the oracle, the histogram's mass is
    checked in full."""
    p = 4 * groups + 3
    q = 2 if model == ISING else 8
    thr = noisy_thresholds(model, L)
    sample = [0, 1, p // 2, p - 4, p - 1]
    with muca.Muca(model, L, q, p, 5) as g:
        g.set_thresholds(thr)
        H = g.iterate(3)
        E, M = g.produce(2)
        spins = g.get_spins()
    assert int(H.sum()) == 3 * p * L * L
    o = MucaOracle(model, L, q, p, 5, chains=sample)
    o.iterate(3, thr=thr)
    e, m = o.produce(2, thr=thr)
    for k, c in enumerate(sample):
        assert np.array_equal(E[:, c], e[:, k]) and np.array_equal(M[:, c], m[:, k]), c
        assert np.array_equal(spins[c], o.spins[k]), c


@pytest.mark.parametrize("L,kind", [(64, "flat"), (32, "noise"), (64, "zeros"), (12, "steps"), (128, "late"),
                                    (66, "ties")])
def test_update_adds_in_order(muca, L, kind):
    """ln W after an update is the sum of its differences in ascending order, each addition
    rounded to FP64, bit for bit (numpy's cumulative sum adds one after the other).  One
    chain that accepts only dE = 0 samples one bin: no difference changes and no boundary
    correction applies, so the update rebuilds ln W from its differences."""
    nb = L * L + 1
    rng = np.random.default_rng(L)
    b = np.arange(nb)
    lnw = {"flat": -0.25 * (b - nb / 2.0) ** 2 / nb, "noise": rng.normal(0, 1, nb), "zeros": np.zeros(nb),
           "steps": np.where(b % 3 == 0, 0.5, 2.0 ** -40) * b,
           "late": -np.abs(b - nb / 2.0) * 0.7 + rng.normal(0, 0.01, nb),
           "ties": np.cumsum(rng.choice([-1.0, 1.0], nb) * 2.0 ** rng.integers(-54, 3, nb))}[kind]
    acc = weights.accessible(ISING, L)
    lnw = np.where(acc, lnw, 0.0)
    with muca.Muca(ISING, L, 2, 1, 3) as g:
        g.set_lnw(lnw)
        g.set_thresholds(np.zeros((nb, 4), dtype=np.uint32))
        H = g.iterate(1)
        assert np.count_nonzero(H) == 1
        g.update_weights()
        got = g.get_lnw()
    v = lnw[acc]
    total = np.cumsum(np.concatenate([[0.0], v[1:] - v[:-1]]))
    want = np.zeros(nb)
    want[acc] = total - total.max()
    assert np.array_equal(got, want)
