"""The FP64 contractions (L <= 384: one task per scale or l range and tile; above:
the eighth-domain kernel) at the edges of their 32-blocks, at the line between
them and for every N: analysis rows against the oracle's Eq. (20) and synthesis
of random coefficients against its Eqs. (32)-(41) within the 1e-11 of FP64
transforms, and a batch over both sides of the line against the single calls."""
import numpy as np
import pytest

import oracle as O
from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian, w_random
from tests.gpu_helpers import relerr, run_analysis, run_synthesis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,lam,J0", [(2, 1, 2.0, 0), (9, 8, 2.0, 1), (31, 2, 2.0, 0), (32, 3, 1.5, 0), (33, 4, 2.0, 2),
                                        (63, 7, 3.0, 0), (65, 6, 2.0, 4), (97, 5, 2.0, 0), (255, 1, 2.0, 3), (256, 8, 2.0, 0),
                                        (257, 2, 2.0, 0), (384, 2, 2.0, 5), (385, 2, 2.0, 5), (512, 2, 2.0, 6), (513, 1, 2.0, 5)])
def test_fp64_contraction(L, N, lam, J0):
    f = flm_gaussian(L, 41, "unit")
    kern = O.kernels(L, N, lam, J0)
    p = B.Plan(L, N, lam, J0, "fp64")
    try:
        W, Wphi = run_analysis(p, f)
        rows = [0, L // 2, 2 * L - 1]
        Wo, Wpo, _ = O.analysis_rows(f, L, N, lam, J0, rows, kern)
        for j in range(p.nscale):
            assert relerr(W[j][:, rows, :], Wo[j]) < 1e-11, j
        assert relerr(Wphi[rows, :], Wpo) < 1e-11
        assert relerr(run_synthesis(p, W, Wphi), f) < 1e-11
        if L <= 97:
            Wr, Wpr = w_random(L, N, p.nscale, 6)
            assert relerr(run_synthesis(p, Wr, Wpr), O.synthesis(Wr, Wpr, L, N, lam, J0, kern)) < 1e-11
    finally:
        p.close()


def test_fp64_batch_over_both_kernels():
    import torch
    plans = [B.Plan(L, N, 2.0, 1, "fp64") for L, N in [(100, 3), (300, 3), (40, 3), (384, 2), (385, 2)]]
    fs = [torch.from_numpy(flm_gaussian(p.L, 60 + i, "cl")).cuda() for i, p in enumerate(plans)]
    Wb, fb = [p.alloc_w() for p in plans], [p.alloc_flm() for p in plans]
    hs = [p.handle for p in plans]
    B.s2dw_analysis_batch(hs, fs, [w[0] for w in Wb], [w[1] for w in Wb])
    B.s2dw_synthesis_batch(hs, [w[0] for w in Wb], [w[1] for w in Wb], fb)
    for p, f, w, g in zip(plans, fs, Wb, fb):
        W, Wp = p.alloc_w()
        h = p.alloc_flm()
        p.analysis(f, W, Wp)
        p.synthesis(w[0], w[1], h)
        assert torch.equal(W, w[0]) and torch.equal(Wp, w[1]) and torch.equal(g, h)
        p.close()
