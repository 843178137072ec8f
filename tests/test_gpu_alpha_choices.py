"""Choice values of the alpha sums on scales that run split matrix products by
default (value 3): 1 and 2 run the chirp-z and the segmented chirp-z that they
name, 3 the products, each agreeing with the FP64 plan at FP32 level (5e-6, as
the tests of the products), and 3 is refused where no products were built."""
import numpy as np
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian
from tests.gpu_helpers import relerr, run_analysis, run_synthesis
from tests.test_gpu_launches import _kernels_of

pytestmark = pytest.mark.gpu


def _scales(p, W):
    out = []
    for j in range(p.nscale):
        _, off, n = p.grids[j]
        out.append(W[off:off + n] if p.multires else W[j])
    return out


@pytest.mark.parametrize("L,N,kw", [(256, 2, {}), (300, 3, {}), (301, 1, {"mw": True}), (400, 2, {"multires": True})])
def test_values_run_as_named(L, N, kw):
    f = flm_gaussian(L, 11, "cl")
    p, p64 = B.Plan(L, N, 2.0, 0, "mixed", **kw), B.Plan(L, N, 2.0, 0, "fp64", **kw)
    try:
        base = p.choices()
        W6, P6 = run_analysis(p64, f)
        default = [i for i in range(2, len(base) - 1) if base[i] == 3]
        assert default
        seen = set()
        for v, names in ((1, "k_czt_alpha"), (2, "_seg"), (3, "k_split_gemm")):
            ch = list(base)
            for i in default:
                ch[i] = v
                try:
                    p.set_choices(ch)
                except B.S2dwError as e:  # no segmented form of this scale
                    assert v == 2 and e.status == B.S2DW_EINVAL
                    ch[i] = 3
            if v not in ch[2:-1]:
                continue
            p.set_choices(ch)
            assert p.choices() == ch
            W, P = run_analysis(p, f)
            for a, b in zip(_scales(p, W), _scales(p, W6)):
                if np.abs(b).max() > 0:
                    assert relerr(a, b) < 5e-6
            g = run_synthesis(p, W6, P6)
            assert relerr(g, f) < 5e-6
            kernels = _kernels_of(lambda: (run_analysis(p, f), run_synthesis(p, W6, P6)))
            ours = [k for k in kernels if "s2dw" in k]
            if ours:
                assert any(names in k and "beta" not in k for k in ours), (v, ours)
                if 3 not in ch[2:-1]:  # (modes 2 and 3 of the products: alpha)
                    assert not any("k_split_gemm<2" in k or "k_split_gemm<3" in k or
                                   "k_split_gemm<(int)2" in k or "k_split_gemm<(int)3" in k for k in ours), (v, ours)
            seen.add(v)
        assert {1, 3} <= seen
    finally:
        p.close()
        p64.close()
    assert B.s2dw_wait_timeouts() == 0


def test_a_segmented_form_is_selected_somewhere():
    p = B.Plan(512, 3, 2.0, 0, "mixed")
    try:
        ch = p.choices()
        both = [j for j in range(p.nscale) if ch[2 + 2 * j] == 3 and p.alpha_method(j, 0)[0] == 2]
        assert both
        for j in both:
            ch[2 + 2 * j] = ch[3 + 2 * j] = 2
        p.set_choices(ch)
        assert [p.alpha_method(j, 1)[0] for j in both] == [2] * len(both)
    finally:
        p.close()


@pytest.mark.parametrize("L,prec", [(64, "mixed"), (256, "fp64")])
def test_products_are_refused_where_not_built(L, prec):
    p = B.Plan(L, 2, 2.0, 0, prec)
    try:
        ch = p.choices()
        assert 3 not in ch[2:-1]
        bad = list(ch)
        bad[2] = 3
        with pytest.raises(B.S2dwError) as e:
            p.set_choices(bad)
        assert e.value.status == B.S2DW_EINVAL and p.choices() == ch
    finally:
        p.close()
