"""The norm of the accuracy check: every element of C_q goes into it as an FP32 value. A sector with one element that counts makes the estimate a formula."""
import math

import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu

# FP32 values whose last bits all count: 1 + 2^-20 less or more a few units of 2^-23
VALUES = [1.0 + 7 * 2.0 ** -23, 1.5 + 2.0 ** -20 - 2.0 ** -23, 2.0 - 2.0 ** -23, 2.0 - 2.0 ** -24 - 2.0 ** -30]


@pytest.mark.parametrize("x", VALUES)
@pytest.mark.parametrize("rows", [(0.0,), (30.0, 0.0), (100.0, 0.0)])   # exponents below the element's
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_estimate_of_one_element(x, rows, sign):
    """est = eta sqrt(4^e) / |c| with the scales' exponents e = 2 of either operand (both
    in [1, 2)): 16 eta / c. The other rows lie 2^-30 below (conversions by FP64 addition and
    by integers) or 2^-100 (general conversion). Bound: the value in FP32 is off by 2^-24 at
    most; its square and a factor by 2^-24 each, which the root halves: 2^-23."""
    import torch
    from paper_2405_12196_gb300 import ytn
    t = [(0,)]
    M = len(rows)
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [1])], (0,), 1)
    B = W.random_tensor((0,), [W.Leg(1, t, [1]), W.Leg(-1, t, [1])], (0,), 2)
    a = np.array([1.0 * 2.0 ** -e for e in rows[:-1]] + [sign * x])
    ctx = ytn.ytn_ctx_create(0)
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    ws = torch.empty(ytn.ytn_workspace_size(plan, ytn.YTN_SPLIT_BF16, 1e-10), dtype=torch.uint8, device=device())
    c = torch.empty(M, dtype=torch.float64, device=device())
    ytn.ytn_tensordot(plan, to_dev(a), to_dev(np.array([1.0])), c, prec=ytn.YTN_SPLIT_BF16, rtol=1e-10, workspace=ws)
    ytn.ytn_sync(ctx)
    assert c[-1].item() == sign * x
    rep = ytn.ytn_tensordot_report(plan, ws)
    s = rep["slices"]
    eta = 2.0 ** (-8 * s - 1) + 2.0 ** -43
    want = 16.0 * eta / x
    assert math.fabs(rep["max_sector_est"] - want) <= 2.0 ** -23 * want
