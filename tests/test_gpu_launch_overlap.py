"""Calls whose launches overlap the end of the kernel before (programmatic stream
serialization) keep stream order: back-to-back calls with other work on the same
buffers between them, and captured calls behind a memset and behind a join of two
streams, give the results of synchronised calls bit for bit."""
import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300.inputs import flm_gaussian

pytestmark = pytest.mark.gpu


def _plan(L, N, prec):
    import torch
    p = B.Plan(L, N, 2.0, 0, prec)
    f = torch.from_numpy(flm_gaussian(L, 3, "cl")).to(p.torch_dtypes()[0]).cuda()
    W, Wp = p.alloc_w()
    return p, f, W, Wp, p.alloc_flm()


def _chain(p, f, W, Wp, g, sync):
    """analysis, W scaled in place, synthesis, f replaced by the result; six times"""
    import torch
    x = f.clone()
    for _ in range(6):
        p.analysis(x, W, Wp)
        sync()
        W.mul_(0.5)
        p.synthesis(W, Wp, g)
        sync()
        x.copy_(g)
        W.zero_()
        sync()
    torch.cuda.synchronize()
    return x


@pytest.mark.parametrize("L,N,prec", [(32, 3, "mixed"), (128, 5, "mixed"), (200, 2, "mixed"), (700, 1, "mixed"),
                                      (100, 2, "fp64"), (520, 1, "fp64")])
def test_back_to_back_calls(L, N, prec):
    import torch
    p, f, W, Wp, g = _plan(L, N, prec)
    ref = _chain(p, f, W, Wp, g, torch.cuda.synchronize)
    for _ in range(3):
        assert torch.equal(_chain(p, f, W, Wp, g, lambda: None), ref)
    p.close()


@pytest.mark.parametrize("L,N,prec", [(32, 3, "mixed"), (200, 2, "mixed"), (100, 2, "fp64")])
def test_captured_calls(L, N, prec):
    import torch
    p, f, W, Wp, g = _plan(L, N, prec)
    q, f2, W2, Wp2, g2 = _plan(L, N, prec)
    p.analysis(f, W, Wp)
    p.synthesis(W, Wp, g)
    q.analysis(f2 * 3, W2, Wp2)
    torch.cuda.synchronize()
    ref = [t.clone() for t in (W, Wp, g, W2)]
    x2 = f2 * 3
    s, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        W.zero_()  # a memset before the first kernel
        s2.wait_stream(s)
        with torch.cuda.stream(s2):
            q.analysis(x2, W2, Wp2)
        p.analysis(f, W, Wp)
        s.wait_stream(s2)
        p.synthesis(W, Wp, g)  # behind the join
    for _ in range(3):
        for t in (W, Wp, g, W2):
            t.fill_(7)
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip((W, Wp, g, W2), ref):
            assert torch.equal(a, b)
    p.close()
    q.close()
