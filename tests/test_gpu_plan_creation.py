"""What creating a plan costs on the device: the basis tables of the matrix
products of a grid are built in two launches, whatever number of tables."""
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
