"""Phase timing: both operands' gathers are phases of their own, also where an untimed call
gathers them in one launch; timing changes no result."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,scattered", [("f64", False), ("c128", True)])
def test_phases_of_the_staged_path(dtype, scattered):
    import torch
    from paper_2405_12196_gb300 import ytn
    t = [(0,), (1,)]
    A = W.random_tensor((0,), [W.Leg(1, t, [90, 31]), W.Leg(-1, t, [40, 77])], (0,), 1, dtype=dtype)
    B = W.random_tensor((0,), [W.Leg(1, t, [40, 77]), W.Leg(-1, t, [55, 8])], (0,), 2, dtype=dtype)
    ctx = ytn.ytn_ctx_create(0)
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    ws = torch.empty(ytn.ytn_workspace_size(plan), dtype=torch.uint8, device=device())
    a, b = (to_dev(x["data"].view(np.float64)) for x in (A, B))
    c = torch.empty(plan.out["size"] * (2 if dtype == "c128" else 1), dtype=torch.float64, device=device())
    outs = []
    for timed in (False, True, False):
        ytn.ytn_profile_enable(ctx, timed)
        c.fill_(float("nan"))
        for _ in range(3):
            ytn.ytn_tensordot(plan, a, b, c, workspace=ws)
        ytn.ytn_sync(ctx)
        outs.append(c.cpu().numpy())
        if timed:
            ph = ytn.ytn_profile_read(ctx)
            want = {"gather_a", "gather_b", "gemm"} | ({"scatter"} if scattered else set())
            assert {k for k in ph if k != "dropped"} == want
            assert all(ph[k][0] == 3 and ph[k][1] > 0 for k in want)
    np.testing.assert_array_equal(outs[1], outs[0])
    np.testing.assert_array_equal(outs[2], outs[0])
