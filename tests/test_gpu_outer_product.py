"""Contractions whose sectors all have K <= 2 (their own kernel on the FP64 path)."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _values(n, seed):
    """Normal numbers among zeros of both signs."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(n)
    x[rng.random(n) < 0.3] = 0.0
    x[rng.random(n) < 0.2] = -0.0
    return x


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("dtype", ["f64", "c128"])
def test_zeros_keep_the_sign_of_a_sum_from_zero(ctx, K, dtype):
    """Each element of C is a sum that starts from +0: no product of a zero gives -0. The
    reference takes the same rounded steps (a product of two doubles is rounded once in
    numpy; the second product is added to it unrounded on the GPU, so for K = 2 one of the
    two factors is a power of two)."""
    import torch
    from paper_2405_12196_gb300 import ytn
    M, N, t, w = 70, 133, [(0,)], 2 if dtype == "c128" else 1
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [K])], (0,), 1, dtype=dtype)
    B = W.random_tensor((0,), [W.Leg(1, t, [K]), W.Leg(-1, t, [N])], (0,), 2, dtype=dtype)
    a, b = _values(M * K * w, 5), _values(K * N * w, 6)
    if K == 2:
        b = np.where(b == 0, b, np.copysign(0.5, b))
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    assert plan.info["max_k"] == K
    c = torch.full((M * N * w,), float("nan"), dtype=torch.float64, device=device())
    ws = torch.empty(ytn.ytn_workspace_size(plan), dtype=torch.uint8, device=device())
    ytn.ytn_tensordot(plan, to_dev(a), to_dev(b), c, workspace=ws)
    ytn.ytn_sync(ctx)

    def product(x, y):
        s = np.zeros((M, N))
        for k in range(K):
            s = s + x[:, k:k + 1] * y[k:k + 1]
        return s

    a, b = a.reshape(M, K, w), b.reshape(K, N, w)
    want = product(a[..., 0], b[..., 0])
    if w == 2:
        re = want - product(a[..., 1], b[..., 1])
        im = (0.0 + product(a[..., 0], b[..., 1])) + product(a[..., 1], b[..., 0])
        want = np.stack([re, im], axis=-1)
    got = c.cpu().numpy().reshape(want.shape)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(np.signbit(got), np.signbit(want))
