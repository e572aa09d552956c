"""Draws that equal their threshold, or differ from it only in the bits that the sweep
passes' tables leave out: the 32-bit test decides (u < A accepts).

A tie comes once in 2^31 attempts, so the tables here are made from draws: all entries
are the draw of one site of one chain (a row's first site, its last one, an inner one),
that draw plus one, or the value with the same upper 31 bits.  Every shape of the
sweeps, few and many chains per block, with a histogram and without, against the oracle
bit for bit."""
import numpy as np
import pytest

from oracle import MucaOracle, sampler

pytestmark = pytest.mark.gpu

ISING, POTTS = 0, 1
SEED = (5 << 32) | 99
ITERATE, THERMALIZE = 1, 2

# model, side, chains, chains per block: a side of every lane count and row form, ragged
# ones among them; 32 and more chains per block make blocks of more than six warps
SHAPES = [(ISING, 8, 3, 0), (ISING, 16, 40, 0), (ISING, 24, 3, 0), (ISING, 24, 48, 64), (ISING, 30, 3, 0),
          (ISING, 62, 3, 0), (ISING, 64, 3, 0), (ISING, 64, 26, 32), (ISING, 62, 26, 32), (ISING, 96, 2, 0),
          (ISING, 126, 2, 0), (ISING, 96, 13, 32), (ISING, 130, 2, 0), (ISING, 160, 2, 0), (ISING, 256, 1, 0),
          (ISING, 258, 1, 0), (POTTS, 5, 3, 0), (POTTS, 8, 20, 0), (POTTS, 8, 200, 192), (POTTS, 15, 3, 0),
          (POTTS, 16, 9, 0), (POTTS, 31, 3, 0), (POTTS, 32, 5, 0), (POTTS, 32, 50, 64), (POTTS, 31, 50, 64),
          (POTTS, 47, 3, 0), (POTTS, 64, 3, 0), (POTTS, 127, 1, 0), (POTTS, 128, 2, 0), (POTTS, 131, 1, 0),
          (POTTS, 160, 1, 0)]


@pytest.fixture(scope="module")
def muca():
    import paper_1212_3975_gb300 as m
    from paper_1212_3975_gb300 import build
    build.build()
    return m


def draw(model, chain, phase, site):
    """Acceptance draw of a site in the first sweep of a phase, clamped as the kernels do."""
    group, word = (site >> 2, site & 3) if model == ISING else (site >> 1, 2 * (site & 1))
    ctr = (group, 0, 0, ((SEED >> 32) << 2) | phase)
    return min(sampler.philox4x32_10(ctr, (SEED & 0xFFFFFFFF, chain))[word], 0xFFFFFFFE)


@pytest.mark.parametrize("model,L,p,cpb", SHAPES)
def test_ties_bit_exact(muca, model, L, p, cpb):
    q = 2 if model == ISING else 8
    rng = np.random.default_rng(1000 * L + p)
    sites = [0, L - 1] + [L * int(rng.integers(1, L)) + x for x in (0, 0, L - 1, L - 1, int(rng.integers(1, L - 1)))]
    with muca.Muca(model, L, q, p, SEED, chains_per_block=cpb) as g:
        n_bins, n_de = g.n_bins, g.n_de
        for site in sites:
            chain = int(rng.integers(0, p))
            for phase in (ITERATE, THERMALIZE):
                u = draw(model, chain, phase, site)
                for A in (u, u + 1, u ^ 1):
                    thr = np.full((n_bins, n_de), A, dtype=np.uint32)
                    g.reset(SEED)
                    g.set_thresholds(thr)
                    sample = sorted({chain, 0, p - 1})
                    o = MucaOracle(model, L, q, p, SEED, chains=sample)
                    if phase == ITERATE:
                        H = g.iterate(1)
                        assert int(H.sum()) == p * L * L
                        o.iterate(1, thr=thr)
                    else:
                        g.thermalize(1)
                        o.thermalize(1, thr=thr)
                    E, M = g.get_energies()
                    spins = g.get_spins()
                    where = (site, chain, phase, A - u)
                    assert np.array_equal(spins[sample], o.spins), where
                    assert np.array_equal(E[sample], o.E) and np.array_equal(M[sample], o.M), where
