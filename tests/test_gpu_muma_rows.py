"""Multimagnetic sweeps on rows of one to three words, full and ragged, against the oracle
bit for bit (iteration, thermalisation, records; tables of noisy weights)."""
import numpy as np
import pytest

from test_gpu_muma import BETA, ISING, random_m_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,p", [(4, 130), (30, 3), (32, 3), (62, 2), (64, 3), (66, 2), (96, 2), (130, 1)])
def test_rows_of_words_bit_exact(L, p):
    import paper_1212_3975_gb300 as muca
    from oracle import MucaOracle, weights
    thr = weights.thresholds_muma(L, random_m_weights(L, L), BETA)
    with muca.Muca(ISING, L, 2, p, 11, muma_beta=BETA) as g:
        g.set_thresholds(thr)
        H = g.iterate(2)
        g.thermalize(1)
        E_rec, M_rec = g.produce(2)
        spins = g.get_spins()
    o = MucaOracle(ISING, L, 2, p, 11, muma_beta=BETA)
    assert np.array_equal(H, o.iterate(2, thr=thr))
    o.thermalize(1, thr=thr)
    e, m = o.produce(2, thr=thr)
    assert np.array_equal(E_rec, e) and np.array_equal(M_rec, m)
    assert np.array_equal(spins, o.spins)
