"""Direct FP64 alpha sums (L_j <= 32, folded over a <-> n - a) at the edges of
their tiles: samples in groups of 32 and tiles of 128, CTAs of 16 rows (small
grids) to 256 rows (L = 520, N = 8).  Analysis rows against the oracle's Eq. (20)
within the 1e-11 that FP64 transforms keep, the synthesis stage V against a
length-n FFT of the same samples within 1e-12 (sums of n <= 1039 terms)."""
import numpy as np
import pytest

import oracle as O
from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian, w_random
from tests.gpu_helpers import relerr, run_analysis, run_synthesis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N", [(2, 1), (17, 2), (32, 3), (33, 1), (65, 4), (100, 3), (128, 1), (129, 5),
                                 (300, 8), (520, 8)])
def test_direct_fp64(L, N):
    p = B.Plan(L, N, 2.0, 0, "fp64")
    try:
        ds = [j for j in range(p.nscale + 1) if p.alpha_method(j, 0)[0] == 0]
        f = flm_gaussian(L, 31, "unit")
        W, Wphi = run_analysis(p, f)
        rows = sorted({0, 1, L // 2, L - 1, min(2 * L - 1, 8), min(2 * L - 1, 15), min(2 * L - 1, 16), 2 * L - 1})
        Wo, Wpo, _ = O.analysis_rows(f, L, N, 2.0, 0, rows, O.kernels(L, N, 2.0, 0))
        for j in ds:
            got, ref = (Wphi[rows, :], Wpo) if j == p.nscale else (W[j][:, rows, :], Wo[j])
            assert relerr(got, ref) < 1e-11, j
        Wr, Wpr = w_random(L, N, p.nscale, 5)
        run_synthesis(p, Wr, Wpr)
        for j in ds:
            w = Wpr if j == p.nscale else Wr[j]
            V = p.stage(1, j)
            Lj = p.support(j)[1] + 1
            if Lj > 0 and V.size:
                ref = np.fft.rfft(w, axis=-1)[..., :Lj] * (2 * np.pi / (2 * L - 1))
                assert relerr(V.reshape(ref.shape), ref) < 1e-12, j
    finally:
        p.close()
