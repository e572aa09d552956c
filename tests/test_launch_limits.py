"""Sizes of sweep launches, checked on the host over every lattice: 32-bit counts of a
block stay below 2^31 whatever a batch is asked to do, and lattices are staged in shared
memory wherever they fit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import test_gpu_sweep_shapes as shapes
from oracle import MucaOracle, reweight

HERE = os.path.dirname(os.path.abspath(__file__))
ISING, POTTS = 0, 1
SIDES = [(ISING, L) for L in range(4, 1025, 2)] + [(POTTS, L) for L in range(3, 256)]


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1212_3975_gb300 import build as b
    lib = b.build()
    out = str(tmp_path_factory.mktemp("plan") / "plan_probe.so")
    subprocess.run([b.nvcc(), *b.ARCH, *b.COMMON, "-shared", "-o", out, os.path.join(HERE, "plan_probe.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True)
    return ctypes.CDLL(out)


@pytest.fixture(scope="module")
def muca():
    import paper_1212_3975_gb300 as m
    from paper_1212_3975_gb300 import build
    build.build()
    return m


def test_batch_launches_keep_counts_in_32_bits(probe):
    """Every attempt of a work unit of a batch may end in one bin.  (Draw positions and
    passes are counted in 32 bits with sign.)"""
    two = (ctypes.c_int * 2)()
    for model, L in SIDES:
        if L % 4:
            continue
        probe.probe_batch(model, L, 4096, two)
        chains, most = two
        assert chains * L * L * most < 2 ** 31 or most == 1, (model, L)
        for n in (1, 7, most - 1, most, most + 1, 3 * most + 5, 2 ** 31 - 1):
            for split in (1, 2, 64):
                if not 0 < n < 2 ** 31:
                    continue
                k = probe.probe_launches(n, split, most)
                assert 1 <= k <= n and k >= min(split, n)
                assert max(n * (s + 1) // k - n * s // k for s in (0, k // 2, k - 1)) <= most, (model, L, n, split)


def test_staging_is_taken_where_it_fits(probe):
    """Lattices in shared memory: every side whose 32 chains fit beside table and histogram
    (a block holds fewer), and no other; automatic and global staging always."""
    two = (ctypes.c_int * 2)()
    takes = {ISING: set(range(4, 163, 2)) | set(range(204, 227, 2)), POTTS: set(range(3, 77))}
    for model, L in SIDES:
        for p in (1, 40, 4865, 20000):
            for hist in (0, 1):
                for staging in (0, 1, 2):
                    ok = probe.probe_launch(model, L, p, staging, 0, hist, two)
                    assert bool(ok) == (staging != 1 or L in takes[model]), (model, L, p, staging)
                    assert not ok or (0 < two[0] <= 227 * 1024 and two[1] >= 1), (model, L, p, staging)


def test_a_pass_that_gives_up_is_an_error(probe):
    """The status that a sweep leaves when a pass does not settle (which needs a mistake in
    the kernel: no input brings it about)."""
    assert probe.probe_fault(0) == 0
    assert probe.probe_fault(1) == -4


@pytest.mark.parametrize("model,L,per_warp", [(ISING, 8, 32), (ISING, 16, 32), (ISING, 18, 4), (ISING, 30, 4),
                                              (ISING, 64, 2), (ISING, 66, 1), (ISING, 256, 1), (POTTS, 6, 16),
                                              (POTTS, 16, 8), (POTTS, 32, 4), (POTTS, 33, 2), (POTTS, 128, 1)])
def test_chains_per_block_is_the_callers(probe, model, L, per_warp):
    """chains_per_block sets the block: that many chains, or what twelve deciding warps, the
    chains there are and the shared memory allow."""
    two = (ctypes.c_int * 2)()
    for p in (5, 100, 3000, 20000):
        if model == ISING and 16 < L <= 32 and p == 20000:
            per_warp = 32  # (a lane per chain)
        for hist in (0, 1):
            for cpb in (32, 64, 128, 256):
                assert probe.probe_launch(model, L, p, 0, cpb, hist, two)
                groups = min(cpb // per_warp, 12, -(-p // per_warp))
                assert two[1] <= groups * per_warp and two[1] % per_warp == 0
                # (a group takes at most 42 KB: fewer groups only where no other would fit)
                assert two[1] == groups * per_warp or two[0] > (227 - 42) * 1024, (p, hist, cpb)


def test_many_chains_of_small_lattices_take_a_lane_each(probe):
    """Ising sides of 18 to 32: rows at once (four chains per warp) with few chains, a lane
    per chain with many; never in batches or with lattices in global memory."""
    two = (ctypes.c_int * 2)()

    def lanes(p, staging=0):
        assert probe.probe_launch(ISING, L, p, staging, 0, 1, two)
        assert two[0] <= 227 * 1024
        return two[1] > 48  # (twelve warps of four chains)

    for L in range(18, 33, 2):
        assert not lanes(1000) and not lanes(4864), L
        for p in (16384, 40000, 1 << 20):
            assert lanes(p) and lanes(p, 1) and not lanes(p, 2), (L, p)
        probe.probe_batch(ISING, L, 16384, two)
        assert two[0] == 16, L


@pytest.mark.gpu
@pytest.mark.parametrize("L", range(18, 33, 2))
def test_a_lane_per_chain_bit_exact(muca, L):
    """Iterations, thermalisation and records of more chains than fill the GPU's warps once,
    a ragged last warp: every chain against the oracle."""
    p = 16389
    thr = shapes.noisy_thresholds(ISING, L)
    with muca.Muca(ISING, L, 2, p, 21) as g:
        g.set_thresholds(thr)
        H1, H2 = g.iterate(2), g.iterate(1)
        g.thermalize(1)
        E, M = g.produce(2)
        n, s1, s2 = g.get_samples()
        spins = g.get_spins()
    o = MucaOracle(ISING, L, 2, p, 21)
    assert np.array_equal(H1, o.iterate(2, thr=thr)) and np.array_equal(H2, o.iterate(1, thr=thr))
    o.thermalize(1, thr=thr)
    e, m = o.produce(2, thr=thr)
    assert np.array_equal(E, e) and np.array_equal(M, m)
    for x, y in zip((n, s1, s2), reweight.bin_series(ISING, L, e, m)):
        assert np.array_equal(x, y)
    assert np.array_equal(spins, o.spins)


@pytest.mark.gpu
def test_batch_counts_all_attempts_of_a_cold_lattice(muca):
    """128 chains of a 4 x 4 lattice that stay in the ground state: more than 2^32 counts of
    one bin by one work unit, in one iteration."""
    n, p = 4194303, 128
    with muca.Muca(ISING, 4, 2, 1, 1) as g:
        nb = g.n_bins
    b = muca.MucaBatch([(ISING, 4, 2, p, 9)])
    b.job(0).set_lnw(-3.0 * (4.0 * np.arange(nb) - 32.0))
    b.iterate(1, n)
    H = b.job(0).get_histogram()
    b.close()
    assert int(H.sum()) == n * p * 16
    assert int(H.max()) > 2 ** 32


@pytest.mark.gpu
@pytest.mark.parametrize("model,L", [(ISING, 4), (ISING, 20), (ISING, 66), (ISING, 162), (ISING, 226), (POTTS, 7),
                                     (POTTS, 33), (POTTS, 70), (POTTS, 75), (POTTS, 76)])
def test_lattices_in_shared_memory_bit_exact(muca, model, L):
    shapes.test_every_shape_bit_exact(muca, model, L, 1)


@pytest.mark.gpu
def test_batch_thermalisation_beyond_one_launch(muca):
    """Intermediate thermalisation is cut into launches by its own length (the iterations
    around it are short), and continues like a single context's."""
    job = (ISING, 4, 2, 40, 3)

    def run(therm):
        b = muca.MucaBatch([job])
        before = muca.kernel_launches()
        b.converge(5, 2, therm_sweeps=therm)
        launches = muca.kernel_launches() - before
        spins, lnw = b.job(0).get_spins(), b.job(0).get_lnw()
        b.close()
        return launches, spins, lnw

    few = run(10)[0]
    launches, spins, lnw = run(900000)   # 128 chains x 16 sites x 900000 sweeps: two launches
    assert launches == few + 1
    with muca.Muca(*job) as g:
        g.converge(5, 2, therm_sweeps=900000)
        assert np.array_equal(g.get_spins(), spins) and np.array_equal(g.get_lnw(), lnw)
