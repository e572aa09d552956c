"""Reweighting where its kernels take different paths, against the oracle's FP64 form:
beta counts of one, a ragged tile and more tiles than two per SM (a setup of half the
threads), FP64 tiles whose weights are products of powers and tiles whose betas lie too
far apart for them, windows of one chunk and of many.  Bounds: FP64 1e-10, FP32 1e-6
relative per observable (C and chi absolutely below 1e-12)."""
import numpy as np
import pytest

import workloads
from oracle import reweight

pytestmark = pytest.mark.gpu

BOUNDS = {"fp64": 1e-10, "fp32": 1e-6}
I, P = workloads.ISING, workloads.POTTS


@pytest.mark.parametrize("model,L,betas", [
    (I, 16, np.array([0.44])),
    (I, 16, np.linspace(0.3, 0.6, 2601)),
    (I, 64, np.concatenate([np.linspace(0.3, 0.5, 24), np.linspace(0.5, 0.52, 15)])),
    (I, 64, np.linspace(-0.2, 0.9, 9)),
    (I, 128, np.linspace(0.40, 0.45, 17)),
    (P, 31, np.linspace(1.2, 1.4, 11)),
    (P, 31, np.array([0.2, 1.3, 2.4])),
    (P, 96, np.linspace(1.30, 1.37, 8))])
def test_reweight_paths(model, L, betas):
    import paper_1212_3975_gb300 as m
    q = 2 if model == I else 8
    n, s1, s2, lnw = workloads.synthetic_samples(model, L, "flat", 2000000, 41)
    ref = reweight.reweight_binned(model, L, q, lnw, n, s1, s2, betas)
    with m.Muca(model, L, q, 8, 1) as g:
        g.set_lnw(lnw)
        g.set_samples(n, s1, s2)
        for prec, bound in BOUNDS.items():
            r = g.reweight(betas, prec)
            for k in ("e", "C", "absm", "chi"):
                scale = np.maximum(np.abs(ref[k]), 1e-12 if k in ("C", "chi") else 1e-300)
                rel = np.abs(r[k] - ref[k]) / scale
                assert rel.max() <= bound, (prec, k, float(rel.max()))
