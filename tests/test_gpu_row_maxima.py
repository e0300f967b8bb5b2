"""The row maxima of the fused slicing against the staged path's (operands in page-locked
host memory): same scale exponents, so the same bits of C. Both kernels (the item count
decides), ragged rows and K."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, run_tensordot

pytestmark = pytest.mark.gpu

RTOL = 1e-10


def _pair(M, K, N):
    t = [(0,)]
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [K])], (0,), M)
    B = W.random_tensor((0,), [W.Leg(1, t, [K]), W.Leg(-1, t, [N])], (0,), N + 1)
    rng = np.random.default_rng(K)
    for rec, rows, first in ((A, M, True), (B, N, False)):
        x = rec["data"].reshape(rows, K) if first else rec["data"].reshape(K, rows).T
        top = rng.integers(0, K, rows)   # where each row's largest lies; some in the last column
        top[::3] = K - 1
        x[np.arange(rows), top] = np.ldexp(1.5, rng.integers(1, 9, rows))
    return A, B


# the last one has 12,288 work items, beyond the line between the kernels
@pytest.mark.parametrize("dims", [(1, 1, 1), (32, 96, 33), (33, 128, 32), (96, 129, 31), (127, 160, 64),
                                  (128, 255, 129), (8190, 3000, 8190)])
def test_fused_row_maxima_match_staged(dims):
    import torch
    from paper_2405_12196_gb300 import ytn
    fresh = ytn.ytn_ctx_create(0)   # its first call leaves the fused variant's result
    A, B = _pair(*dims)
    plan, got, res = run_tensordot(fresh, A, B, (1,), (0,), prec=ytn.YTN_SPLIT_BF16, rtol=RTOL)
    assert plan.info["split_fused"] == 1 and res["split_variant"] == 1
    a, b = (torch.from_numpy(x["data"]).pin_memory() for x in (A, B))
    c = torch.full((plan.out["size"],), float("nan"), dtype=torch.float64, device=device())
    ws = torch.empty(ytn.ytn_workspace_size(plan, ytn.YTN_SPLIT_BF16, RTOL), dtype=torch.uint8, device=device())
    staged = ytn.ytn_tensordot(plan, a, b, c, prec=ytn.YTN_SPLIT_BF16, rtol=RTOL, workspace=ws)
    ytn.ytn_sync(fresh)
    assert staged["split_variant"] == 0
    np.testing.assert_array_equal(c.cpu().numpy(), got["data"])
