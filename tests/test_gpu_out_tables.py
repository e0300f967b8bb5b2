"""The tables by which the GEMMs write C's blocks are kept only where they are small beside C
(or below 1 MiB): products with a long thin side go through the dense matrix and the scatter,
which the phase record shows, with the same results."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu


def _pair(rows, K, cols):
    r, c = (W.Leg(1, [(q,) for q in range(len(d))], d) for d in (rows, cols))
    k = W.Leg(1, [(q,) for q in range(max(len(rows), len(cols)))], [K] * max(len(rows), len(cols)))
    A = W.random_tensor((0,), [r, k.conj()], (0,), 1)
    B = W.random_tensor((0,), [k, c.conj()], (0,), 2)
    return A, B


@pytest.mark.parametrize("prec", ["YTN_FP64", "YTN_SPLIT_BF16"])
@pytest.mark.parametrize("rows,K,cols,scattered", [([200000], 2, [3], True), ([3], 2, [120000], True),
                                                   ([150001, 5], 7, [2, 9], True), ([70000, 900], 3, [1, 2], False),
                                                   ([9000, 30], 5, [700, 2000], False)])
def test_long_thin_products_keep_no_tables(prec, rows, K, cols, scattered):
    import torch
    from paper_2405_12196_gb300 import ytn
    prec, rtol = getattr(ytn, prec), 1e-10
    A, B = _pair(rows, K, cols)
    ctx = ytn.ytn_ctx_create(0)
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    ws = torch.empty(ytn.ytn_workspace_size(plan, prec, rtol), dtype=torch.uint8, device=device())
    c = torch.full((plan.out["size"],), float("nan"), dtype=torch.float64, device=device())
    a, b = to_dev(A["data"]), to_dev(B["data"])
    ytn.ytn_tensordot(plan, a, b, c, prec=prec, rtol=rtol, workspace=ws)
    ytn.ytn_profile_enable(ctx, True)
    c.fill_(float("nan"))
    ytn.ytn_tensordot(plan, a, b, c, prec=prec, rtol=rtol, workspace=ws)
    phases = ytn.ytn_profile_read(ctx)
    assert ("scatter" in phases) == scattered
    got, at, a0, b0 = c.cpu().numpy(), 0, 0, 0
    for m, n in zip(rows, cols):
        x, y = A["data"][a0:a0 + m * K].reshape(m, K), B["data"][b0:b0 + K * n].reshape(K, n)
        want = x @ y
        err = np.linalg.norm(got[at:at + m * n].reshape(m, n) - want)
        assert err <= (1e-15 * K if prec == ytn.YTN_FP64 else rtol) * np.linalg.norm(want)
        a0, b0, at = a0 + m * K, b0 + K * n, at + m * n
