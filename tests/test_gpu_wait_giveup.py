"""Give-up path of the bounded waits inside the kernels: with waits that end at
once the products, direct sums and contractions of a plan stop in every role, are
counted, and leave tensor memory, barriers and context in order: the same plan
then transforms as before, and waits of ordinary length count nothing."""
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian

pytestmark = pytest.mark.gpu


def _roundtrip(p, f):
    import torch
    W, Wp = p.alloc_w()
    p.analysis(f, W, Wp)
    g = p.alloc_flm()
    p.synthesis(W, Wp, g)
    torch.cuda.synchronize()
    return W, Wp, g


@pytest.mark.parametrize("L,N,kw", [(32, 2, {}), (200, 2, {}), (361, 5, {}), (300, 3, {"mw": True}),
                                    (512, 1, {}), (512, 5, {}), (512, 8, {})])
def test_kernels_give_up_in_every_role(L, N, kw):
    import torch
    f = torch.from_numpy(flm_gaussian(L, 3, "cl")).to(torch.complex64).cuda()
    p = B.Plan(L, N, 2.0, 0, "mixed", **kw)
    try:
        before = [t.clone() for t in _roundtrip(p, f)]
        assert B.s2dw_wait_timeouts() == 0
        for limit in (0, 50, 1500):  # cycles: less than a bulk copy takes, up to about as long
            B.s2dw_plan_wait_probe(p.handle, limit)
            n = B.s2dw_wait_timeouts()  # synchronises: the launches have ended
            # (at L = 32 only the direct alpha sums have such waits; they look once, suspended, before a limit ends them)
            assert n > 0 or limit > (0 if L == 32 else 50)
        B.s2dw_plan_wait_probe(p.handle, 2_000_000_000)
        assert B.s2dw_wait_timeouts() == 0
        for a, b in zip(before, _roundtrip(p, f)):
            assert torch.equal(a, b)
        assert B.s2dw_wait_timeouts() == 0
    finally:
        p.close()


def test_fp64_plans_have_no_such_waits():
    p = B.Plan(40, 2, 2.0, 0, "fp64")
    try:
        with pytest.raises(B.S2dwError) as e:
            B.s2dw_plan_wait_probe(p.handle, 1000)
        assert e.value.status == B.S2DW_ENOTSUP
    finally:
        p.close()
