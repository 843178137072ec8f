"""Magnitudes near the top of FP32 through the split matrix products: the sums
carry no scale of the basis, so they stay finite as long as the transforms'
own sums do (the scales are powers of two: the relative error is that of any
other magnitude, 5e-6 as in the tests of the products' tiles)."""
import numpy as np
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian
from tests.gpu_helpers import relerr, run_analysis, run_synthesis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,kw", [(150, 2, {}), (200, 1, {}), (200, 3, {"mw": True}), (256, 2, {})])
@pytest.mark.parametrize("amp", [1e33, 1e35])
def test_products_near_the_top_of_fp32(L, N, kw, amp):
    f = flm_gaussian(L, 23, "cl") * amp
    pm, p64 = B.Plan(L, N, 2.0, 0, "mixed", **kw), B.Plan(L, N, 2.0, 0, "fp64", **kw)
    try:
        Wm, Pm = run_analysis(pm, f)
        W6, P6 = run_analysis(p64, f)
        assert np.isfinite(Wm).all() and np.isfinite(Pm).all()
        for j in range(pm.nscale):
            if np.abs(W6[j]).max() > 0:
                assert relerr(Wm[j], W6[j]) < 5e-6, j
        g = run_synthesis(pm, W6, P6)
        assert np.isfinite(g).all()
        assert relerr(g, f) < 5e-6
    finally:
        pm.close()
        p64.close()
    assert B.s2dw_wait_timeouts() == 0
