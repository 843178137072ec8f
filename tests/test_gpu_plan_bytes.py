"""The workspace bound against the workspaces of plans of random configurations."""
import math
import random

import pytest

from paper_1308_5706_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(4))
def test_bound_covers_random_plans(seed):
    rng = random.Random(seed)
    for _ in range(30):
        prec = rng.choice(["mixed", "mixed", "fp64"])
        L = int(round(math.exp(rng.uniform(math.log(2), math.log(2048 if prec == "mixed" else 700)))))
        N, lam = min(L, rng.randint(1, 8)), rng.choice([1.3, 1.6, 2.0, 2.0, 3.0])
        grid = rng.choice([0, 0, B.S2DW_MULTIRES, B.S2DW_MW])
        J0 = rng.randint(0, 2 if lam > 1.4 else 1)
        kw = {"multires": grid == B.S2DW_MULTIRES, "mw": grid == B.S2DW_MW}
        flags = (B.S2DW_MIXED if prec == "mixed" else B.S2DW_FP64) | B.S2DW_REAL_SIGNAL | grid
        try:
            p = B.Plan(L, N, lam, J0, prec, **kw)
        except B.S2dwError as e:
            assert e.status in (B.S2DW_EINVAL, B.S2DW_ENOTSUP)
            continue
        ws = p.info["workspace_bytes"]
        p.close()
        b = B.s2dw_plan_bytes(L, N, lam, J0, flags)
        assert ws <= b <= 1.5 * ws + (8 << 20), (L, N, lam, J0, prec, kw, ws, b)
