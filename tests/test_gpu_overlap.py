"""C in an operand's own buffer. The first call on a plan is the one that picks the path
by running several: each of them must see the operands, not the last one's result."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu

RTOL = 1e-10


def _pair(M, K, N):
    t = [(0,)]
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [K])], (0,), 21)
    B = W.random_tensor((0,), [W.Leg(1, t, [K]), W.Leg(-1, t, [N])], (0,), 22)
    return A, B


@pytest.mark.parametrize("prec", ["YTN_FP64", "YTN_SPLIT_BF16", "YTN_AUTO"])
@pytest.mark.parametrize("into,shift", [("A", 0), ("B", 0), ("A", 101), ("B", -64)])
def test_first_call_with_c_over_an_operand(prec, into, shift):
    import torch
    from paper_2405_12196_gb300 import ytn
    prec = getattr(ytn, prec)
    M, K, N = 200, 170, 190
    A, B = _pair(M, K, N)
    want = A["data"].reshape(M, K) @ B["data"].reshape(K, N)
    fresh = ytn.ytn_ctx_create(0)   # no choice of an earlier call
    plan = ytn.ytn_plan(fresh, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    ws = torch.empty(ytn.ytn_workspace_size(plan, prec, RTOL), dtype=torch.uint8, device=device())
    mem = torch.zeros(3 * max(M * K, K * N, M * N), dtype=torch.float64, device=device())
    at = mem.numel() // 3
    src = A if into == "A" else B
    op = mem[at:at + src["data"].size]
    op.copy_(to_dev(src["data"]))
    c = mem[at + shift:at + shift + M * N]
    other = to_dev((B if into == "A" else A)["data"])
    a, b = (op, other) if into == "A" else (other, op)
    ytn.ytn_tensordot(plan, a, b, c, prec=prec, rtol=RTOL, workspace=ws)
    ytn.ytn_sync(fresh)
    got = c.cpu().numpy().reshape(M, N)
    assert np.linalg.norm(got - want) <= RTOL * np.linalg.norm(want)
    # the choices are still open, and the next call with C apart makes them
    if prec == ytn.YTN_FP64:
        return
    assert ytn.ytn_plan_tuning(plan, 5)["split_variant"] == -1
    a2, b2, c2 = to_dev(A["data"]), to_dev(B["data"]), torch.empty(M * N, dtype=torch.float64, device=device())
    ytn.ytn_tensordot(plan, a2, b2, c2, prec=prec, rtol=RTOL, workspace=ws)
    ytn.ytn_sync(fresh)
    assert ytn.ytn_plan_tuning(plan, 5)["split_variant"] in (0, 1)
    np.testing.assert_allclose(c2.cpu().numpy().reshape(M, N), want, rtol=0, atol=RTOL * np.linalg.norm(want))
