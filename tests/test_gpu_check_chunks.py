"""The accuracy check of sectors whose rows span several CTAs (4096 rows of A and B
together each): the estimate, the flagged sectors and the order of the sums."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import device, to_dev

pytestmark = pytest.mark.gpu

RTOL = 1e-10


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _sectors(dims, make, seed=3):
    """One U(1) sector per (M, K, N); make(q, rng, M, K, N) gives its two matrices."""
    q = [(i,) for i in range(len(dims))]
    M, K, N = ([d[i] for d in dims] for i in range(3))
    A = W.random_tensor((0,), [W.Leg(1, q, M), W.Leg(-1, q, K)], (0,), seed)
    B = W.random_tensor((0,), [W.Leg(1, q, K), W.Leg(-1, q, N)], (0,), seed + 1)
    rng = np.random.default_rng(seed)
    mats = [make(i, rng, *d) for i, d in enumerate(dims)]
    A["data"] = np.concatenate([a.reshape(-1) for a, _ in mats])
    B["data"] = np.concatenate([b.reshape(-1) for _, b in mats])
    return A, B, mats


def _run(ctx, A, B):
    import torch
    from paper_2405_12196_gb300 import ytn
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    ws = torch.empty(ytn.ytn_workspace_size(plan, ytn.YTN_SPLIT_BF16, RTOL), dtype=torch.uint8, device=device())
    c = torch.full((plan.out["size"],), float("nan"), dtype=torch.float64, device=device())
    a, b = to_dev(A["data"]), to_dev(B["data"])

    def call():
        ytn.ytn_tensordot(plan, a, b, c, prec=ytn.YTN_SPLIT_BF16, rtol=RTOL, workspace=ws)
        ytn.ytn_sync(ctx)
        return c.cpu().numpy(), ytn.ytn_tensordot_report(plan, ws)
    return call


def _scales(x):
    """Sum of 4^e over the rows, e = 2 + floor(log2 max)."""
    m = np.abs(x).max(axis=1)
    e = np.frexp(m)[1] + 1
    return np.where(m > 0, 4.0 ** e, 0.0).sum()


# sectors of one chunk and of several, chunks that hold rows of both operands
@pytest.mark.parametrize("dims", [[(4000, 3, 90)], [(4096, 2, 1)], [(5, 2, 4099)], [(4097, 5, 8200), (3, 4, 2), (2000, 9, 2100)],
                                  [(40001, 2, 7), (20, 3, 30), (9, 2, 24999)]])
def test_estimate_over_chunks(ctx, dims):
    """est_q = eta sqrt(K sum 4^e sum 4^f) / |C_q|. Bound: the norm is summed in FP32, at
    most 32 + 5 additions of 2^-24 in a warp and one atomic addition per warp's 32 x 32
    elements."""
    def make(i, rng, M, K, N):
        a, b = rng.standard_normal((M, K)), rng.standard_normal((K, N))
        return a * 2.0 ** rng.integers(-6, 7, (M, 1)), b * 2.0 ** rng.integers(-6, 7, (1, N))
    A, B, mats = _sectors(dims, make)
    _, rep = _run(ctx, A, B)()
    eta = 2.0 ** (-8 * rep["slices"] - 1) + 2.0 ** -43
    est = [eta * np.sqrt(a.shape[1] * _scales(a) * _scales(b.T)) / np.linalg.norm(a @ b) for a, b in mats]
    adds = 40 + max((d[0] / 32 + 8) * (d[2] / 32 + 8) for d in dims)
    assert abs(rep["max_sector_est"] - max(est)) <= adds * 2.0 ** -24 * max(est)


def test_flagged_sectors_of_several_chunks(ctx):
    """Sectors whose products cancel are recomputed in FP64, wherever they stand among those
    that do not and however many chunks they have."""
    dims = [(20, 9, 30), (9000, 4, 500), (4200, 4, 4100), (8, 6, 70), (4097, 2, 3), (5000, 6, 90)]

    def make(i, rng, M, K, N):
        a, b = rng.standard_normal((M, K)), rng.standard_normal((K, N))
        if i % 2 == 0:   # the second half of K nearly takes back what the first gives
            h = K // 2
            a[:, h:2 * h] = -a[:, :h]
            b[h:2 * h] = b[:h] * (1 + 1e-9 * rng.standard_normal((h, N)))
            a[:, 2 * h:] = 0
        return a, b
    A, B, mats = _sectors(dims, make)
    got, rep = _run(ctx, A, B)()
    assert rep["nsectors"] == len(dims) and rep["nfallback"] == len(dims) // 2
    assert rep["fallback_flops"] == sum(2.0 * m * k * n for m, k, n in dims[::2])
    at = 0
    for i, (a, b) in enumerate(mats):
        x = got[at:at + a.shape[0] * b.shape[1]].reshape(a.shape[0], -1)
        at += x.size
        scale = np.abs(a) @ np.abs(b)
        assert np.all(np.abs(x - a @ b) <= (1e-15 if i % 2 == 0 else 1e-10) * (a.shape[1] + 8) * scale.max())


def test_the_scales_are_summed_in_a_fixed_order(ctx):
    """Row scales over 26 binary orders, so that the sum depends on its order; every row but
    one cancels exactly, so that the norm is one addend: the estimate repeats bit for bit."""
    def make(i, rng, M, K, N):
        a = np.ldexp(rng.random((M, 1)) + 1.0, -rng.integers(0, 27, (M, 1)))
        a = np.concatenate([a, -a], axis=1)
        a[M // 2] = (1.0, 0.0)
        return a, np.ones((K, N))
    A, B, _ = _sectors([(400000, 2, 1)], make)
    call = _run(ctx, A, B)
    seen = {call()[1]["max_sector_est"] for _ in range(40)}
    assert len(seen) == 1
