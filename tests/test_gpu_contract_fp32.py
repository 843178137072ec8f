"""The FP32 contractions (direct for small L, tile kernel above): Fourier cube, scaling
part and synthesis against the FP64 plan at the edges of its 32-blocks, of its
ranges (L = 448 | 449 for N <= 2, 384 for N <= 4, 320, 288 for N > 6) and for every N, within the 1e-5 that the mixed path keeps
(FP32 sums of at most L terms); and independence of how a launch cuts its tasks
(rows per thread, l ranges): a job in a large batch equals the job alone."""
import numpy as np
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian, w_random
from tests.gpu_helpers import relerr, run_analysis, run_synthesis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,lam,J0", [(2, 1, 2.0, 0), (9, 8, 2.0, 1), (31, 2, 2.0, 0), (32, 3, 1.5, 0), (33, 4, 2.0, 2),
                                        (63, 7, 3.0, 0), (65, 6, 2.0, 4), (97, 5, 2.0, 0), (193, 1, 2.0, 7),
                                        (448, 2, 2.0, 0), (449, 2, 2.0, 0), (384, 4, 2.0, 0), (385, 4, 2.0, 1),
                                        (320, 5, 2.0, 0), (321, 6, 2.0, 0), (288, 7, 2.0, 1), (289, 8, 2.0, 0),
                                        (640, 3, 2.0, 1), (641, 2, 2.0, 1), (655, 7, 2.0, 0), (672, 8, 3.0, 0),
                                        (705, 6, 1.7, 2), (800, 5, 2.0, 0), (673, 1, 2.0, 0)])
def test_direct_contraction_vs_fp64(L, N, lam, J0):
    f = flm_gaussian(L, 17, "unit")
    pm, p64 = B.Plan(L, N, lam, J0, "mixed"), B.Plan(L, N, lam, J0, "fp64")
    try:
        run_analysis(pm, f)
        run_analysis(p64, f)
        for j in range(pm.nscale + 1):
            ref = p64.stage(0, j)
            if ref.size and np.abs(ref).max() > 0:
                assert relerr(pm.stage(0, j), ref) < 1e-5, j
        Wr, Wpr = w_random(L, N, pm.nscale, 3)
        ref = run_synthesis(p64, Wr, Wpr)
        assert relerr(run_synthesis(pm, Wr, Wpr), ref) < 1e-5
    finally:
        pm.close()
        p64.close()


def test_direct_contraction_task_cut_does_not_enter_results():
    import torch
    plans = [B.Plan(L, N, 2.0, 1, "mixed") for L, N in [(100, 3)] * 20 + [(128, 3), (40, 3), (100, 5)]]
    fs = [torch.from_numpy(flm_gaussian(p.L, 60 + i, "cl")).to(torch.complex64).cuda() for i, p in enumerate(plans)]
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
    for p in plans:
        p.close()
