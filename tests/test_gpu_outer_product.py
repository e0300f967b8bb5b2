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


def _blocks(rows, cols, ks, order, seed=5):
    """Row and column legs of two charges and a small third leg on either side, so that C's
    sectors have several row and column blocks; order: where the contracted leg stands."""
    t = [(0,), (1,)]
    r, c, k = W.Leg(1, t, rows), W.Leg(-1, t, cols), W.Leg(-1, t[:len(ks)], ks)
    x = W.Leg(1, t, [2, 1])
    if order == "last-first":
        A, axa = W.random_tensor((0,), [r, x, k], (0,), seed), (2,)
        B, axb = W.random_tensor((0,), [k.conj(), x.conj(), c], (0,), seed + 1), (0,)
    else:
        A, axa = W.random_tensor((0,), [k, r, x], (0,), seed), (0,)
        B, axb = W.random_tensor((0,), [x.conj(), c, k.conj()], (0,), seed + 1), (2,)
    return A, B, axa, axb


def _drop(T, rng, keep):
    off = np.concatenate([[0], np.cumsum(np.prod(T["D"], axis=1))])
    kept = sorted(rng.choice(len(T["t"]), max(1, int(keep * len(T["t"]))), replace=False).tolist())
    return {**T, "t": T["t"][kept], "D": T["D"][kept], "data": np.concatenate([T["data"][off[i]:off[i + 1]] for i in kept])}


def _against_oracle(ctx, A, B, axa, axb, pinned=False):
    import torch
    from gpu_helpers import FP64_RTOL, check_against_oracle, oracle_tensordot
    from paper_2405_12196_gb300 import ytn
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, axa, axb)
    assert plan.info["max_k"] <= 2
    want = oracle_tensordot(A, B, axa, axb)
    if not plan.out["size"]:
        assert np.asarray(want["data"]).size == 0
        return
    c = torch.full((plan.out["size"],), float("nan"), dtype=torch.float64)
    c = c.pin_memory() if pinned else c.to(device())
    ws = torch.empty(max(256, ytn.ytn_workspace_size(plan)), dtype=torch.uint8, device=device())
    ytn.ytn_tensordot(plan, to_dev(A["data"]), to_dev(B["data"]), c, workspace=ws)
    ytn.ytn_sync(ctx)
    check_against_oracle({**plan.out, "data": c.cpu().numpy()}, want, rtol=FP64_RTOL)


# the kernel's tiles have 64 rows and 128 columns; a sector's are 2 or 3 times the legs' dims
# here, and exactly these with a leg dimension of their own below
@pytest.mark.parametrize("m", [1, 63, 64, 65, 130])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("ks", [(1,), (2,), (1, 2)])
@pytest.mark.parametrize("order", ["last-first", "first-last"])
def test_tile_edges_against_the_oracle(ctx, m, n, ks, order):
    _against_oracle(ctx, *_blocks([m, 3], [2, n], ks, order))


@pytest.mark.parametrize("m", [1, 63, 64, 65, 130])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("order", [(0, 1), (1, 0)])
def test_one_block_sectors(ctx, m, n, order):
    t = [(0,)]
    for K in (1, 2):
        la, lb = [W.Leg(1, t, [m]), W.Leg(-1, t, [K])], [W.Leg(1, t, [K]), W.Leg(-1, t, [n])]
        A = W.random_tensor((0,), [la[i] for i in order], (0,), 3)
        B = W.random_tensor((0,), [lb[i] for i in order], (0,), 4)
        _against_oracle(ctx, A, B, (order.index(1),), (order.index(0),))


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("order", ["last-first", "first-last"])
def test_missing_blocks_and_host_results(ctx, seed, order):
    rng = np.random.default_rng(seed)
    A, B, axa, axb = _blocks([65, 40], [129, 7], (1, 2), order)
    _against_oracle(ctx, A, B, axa, axb, pinned=True)
    A, B = _drop(A, rng, 0.6), _drop(B, rng, 0.6)
    _against_oracle(ctx, A, B, axa, axb, pinned=seed % 2 == 1)
