"""Beta and alpha sums as split FP16 matrix products (mixed plans): W and f_lm
against the FP64 plan at the edges of the 128-wide tiles, the 64-column parity
tiles and the 32-term stages, on the DH, multi-resolution and MW grids, at FP32
level (every operand is held to 2^-24, so sums of up to 2L terms stay within the
5e-6 that FP32 transforms of these sizes keep), and for inputs of any magnitude
(rows are scaled by powers of two)."""
import numpy as np
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian, w_random
from tests.gpu_helpers import relerr, run_analysis, run_synthesis

pytestmark = pytest.mark.gpu


def _compare(L, N, lam, J0, amp=1.0, **kw):
    f = flm_gaussian(L, 23, "cl") * amp
    pm, p64 = B.Plan(L, N, lam, J0, "mixed", **kw), B.Plan(L, N, lam, J0, "fp64", **kw)
    try:
        Wm, Pm = run_analysis(pm, f)
        W6, P6 = run_analysis(p64, f)
        for j in range(pm.nscale):
            _, off, n = pm.grids[j]
            a, b = (Wm[off:off + n], W6[off:off + n]) if kw.get("multires") else (Wm[j], W6[j])
            if np.abs(b).max() > 0:
                assert relerr(a, b) < 5e-6, j
        if np.abs(P6).max() > 0:
            assert relerr(Pm, P6) < 5e-6
        if kw.get("multires"):
            Wr, Wp = W6, P6
        else:
            Wr, Wp = w_random(L, N, pm.nscale, 29, nb=L if kw.get("mw") else 2 * L)
            Wr, Wp = Wr * amp, Wp * amp
        assert relerr(run_synthesis(pm, Wr, Wp), run_synthesis(p64, Wr, Wp)) < 5e-6
    finally:
        pm.close()
        p64.close()
    assert B.s2dw_wait_timeouts() == 0


@pytest.mark.parametrize("L,N,lam,J0,kw", [(113, 1, 2.0, 0, {}), (127, 2, 2.0, 6, {}), (128, 3, 2.0, 0, {}),
                                           (129, 8, 3.0, 0, {}), (191, 4, 1.6, 0, {}), (193, 5, 2.0, 1, {}),
                                           (256, 1, 2.0, 0, {}), (257, 2, 2.0, 3, {}), (300, 2, 2.0, 0, {"multires": True}),
                                           (130, 3, 2.0, 0, {"mw": True}), (255, 1, 2.0, 0, {"mw": True})])
def test_products_match_fp64(L, N, lam, J0, kw):
    _compare(L, N, lam, J0, **kw)


@pytest.mark.parametrize("amp", [1e-30, 1e-12, 1e12, 1e30])
def test_products_take_any_magnitude(amp):
    _compare(150, 2, 2.0, 0, amp)


def test_largest_grid_matches_itself_split():
    """L = 2048 (half-length transforms against products): both forms of the beta
    sums of one plan agree at FP32 level."""
    import torch
    L = 2048
    f = torch.from_numpy(flm_gaussian(L, 7, "cl")).to(torch.complex64).cuda()
    p = B.Plan(L, 1, 2.0, 0, "mixed")
    out = []
    base = p.choices()
    for mode in (1, 0):
        ch = list(base)
        ch[0] = ch[1] = mode
        p.set_choices(ch)
        W, Wp = p.alloc_w()
        g = p.alloc_flm()
        p.analysis(f, W, Wp)
        p.synthesis(W, Wp, g)
        torch.cuda.synchronize()
        out.append((W, g))
    for j in range(p.nscale):
        a, b = out[0][0][j], out[1][0][j]
        ref = float(b.abs().max())
        if ref > 0:
            assert float((a - b).abs().max()) < 5e-6 * ref
    assert float((out[0][1] - out[1][1]).abs().max()) < 5e-6 * float(out[1][1].abs().max())
    p.close()
