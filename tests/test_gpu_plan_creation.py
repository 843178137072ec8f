"""What creating a plan costs on the device: the basis tables of the matrix
products of a grid are built in two launches, those of the direct alpha sums in
one, whatever number of tables, and a
closed plan's workspace stays with the library for the next one (mapping it anew
costs 1 ms per GB) also beside the largest shared tables."""
import pytest

from paper_1308_5706_gb300 import binding as B
from tests.test_gpu_launches import _kernels_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N,kw", [(200, 2, {}), (255, 1, {"mw": True})])
def test_basis_tables_take_two_launches(L, N, kw):
    keep = B.Plan(L, 1, 2.0, 0, "mixed")  # the shared tables exist
    names = _kernels_of(lambda: B.Plan(L, N, 2.0, 0, "mixed", **kw).close())
    keep.close()
    if not names:
        pytest.skip("profiler recorded no CUDA kernels")
    assert len([n for n in names if "k_sg_" in n]) == 2, names
    assert len([n for n in names if "k_tc_basis" in n]) == 1, names


def test_workspace_stays_mapped_beside_the_largest_tables():
    import torch
    big = B.Plan(2048, 1, 2.0, 0, "mixed")
    try:
        p = B.Plan(1024, 5, 2.0, 0, "mixed")
        ws = p.info["workspace_bytes"]
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        p.close()
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        assert after - before < ws // 2
        B.Plan(1024, 5, 2.0, 0, "mixed").close()  # reuses it
        torch.cuda.synchronize()
        assert abs(torch.cuda.mem_get_info()[0] - after) < ws // 2
    finally:
        big.close()


def test_freed_blocks_beyond_the_cache_go_back():
    import torch
    torch.cuda.synchronize()
    ps = [B.Plan(2048, 8, 2.0, 0, "mixed") for _ in range(6)]  # some 28 GB beside the tables
    total = sum(p.info["workspace_bytes"] for p in ps)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for p in ps:
        p.close()
    torch.cuda.synchronize()
    B.Plan(32, 1, 2.0, 0, "mixed").close()  # (the pool gives back at a synchronisation after a free)
    torch.cuda.synchronize()
    freed = torch.cuda.mem_get_info()[0] - before
    assert total > 20 << 30
    assert freed > total - (17 << 30)
