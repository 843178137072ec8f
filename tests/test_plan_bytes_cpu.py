"""Workspace bound of a plan (host only): the statuses of plan creation, and at
least the workspaces measured on the device for plans of every kind of path."""
import os

import pytest

from paper_1308_5706_gb300 import binding as B
from paper_1308_5706_gb300 import serve

pytestmark = pytest.mark.skipif(not os.path.exists(B.LIB_PATH), reason="libs2dw.so not built")

MIXED, FP64 = B.S2DW_MIXED, B.S2DW_FP64


@pytest.mark.parametrize("L,N,flags,measured_mb", [
    (32, 3, MIXED, 0.58), (64, 3, MIXED, 1.28), (128, 5, MIXED, 10.7), (129, 8, MIXED, 41.4), (200, 8, MIXED, 67.4),
    (361, 4, MIXED, 92.8), (361, 8, MIXED, 179.0), (511, 3, MIXED | B.S2DW_MW, 127.4), (723, 6, MIXED, 561.0),
    (900, 8, MIXED, 952.0), (1024, 5, MIXED, 746.7), (1024, 5, MIXED | B.S2DW_MULTIRES, 602.1), (2048, 8, MIXED, 4698.7),
    (64, 3, FP64, 2.08), (256, 3, FP64, 45.3), (512, 3, FP64, 247.8)])
def test_bound_covers_the_plan(L, N, flags, measured_mb):
    b = B.s2dw_plan_bytes(L, N, 2.0, 0, flags | B.S2DW_REAL_SIGNAL)
    assert measured_mb * 1e6 <= b <= 1.25 * measured_mb * 1e6 + 4e6


def test_admission_counts_the_whole_workspace():
    r = serve.Request(0, "analysis", 200, 8, 2.0, 0.0)
    assert serve._workspace_estimate(r, 4) >= 67_400_000  # the plan's workspace_bytes are 67.5e6
    r = serve.Request(0, "analysis", 512, 3, 2.0, 0.0)
    assert serve._workspace_estimate(r, 8) >= 247_800_000


@pytest.mark.parametrize("args,status", [((1, 1, 2.0, 0, MIXED), B.S2DW_EINVAL), ((32, 0, 2.0, 0, MIXED), B.S2DW_EINVAL),
                                         ((32, 3, 1.0, 0, MIXED), B.S2DW_EINVAL), ((32, 3, 2.0, 6, MIXED), B.S2DW_EINVAL),
                                         ((32, 3, 2.0, 0, 0), B.S2DW_EINVAL), ((4096, 3, 2.0, 0, MIXED), B.S2DW_ENOTSUP),
                                         ((32, 9, 2.0, 0, FP64), B.S2DW_ENOTSUP)])
def test_statuses_are_those_of_plan_creation(args, status):
    for call in (B.s2dw_plan_bytes, B.s2dw_plan):
        with pytest.raises(B.S2dwError) as e:
            call(*args)
        assert e.value.status == status
