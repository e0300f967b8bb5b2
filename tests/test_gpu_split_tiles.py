"""The split-precision grouped GEMM at the edges of its tiles (pairs of 128 columns times
128 rows; 64-wide column tails), of its K stages and chunks, of C's blocks, which it
writes itself, and of its conversion to FP64, against the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_against_oracle, device, oracle_tensordot, run_tensordot, to_dev

pytestmark = pytest.mark.gpu

RTOL = 1e-10


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _dense(M, K, N, seed, scale=None):
    t = [(0,)]
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [K])], (0,), seed)
    B = W.random_tensor((0,), [W.Leg(1, t, [K]), W.Leg(-1, t, [N])], (0,), seed + 1)
    return A, B, (1,), (0,)


def _blocks(rows, cols, ks, seed):
    """Row, column and contracted legs of many charges: C has blocks of every shape."""
    r = W.Leg(1, [(q,) for q in range(len(rows))], rows)
    c = W.Leg(-1, [(q,) for q in range(len(cols))], cols)
    k = W.Leg(-1, [(q,) for q in range(len(ks))], ks)
    x = W.Leg(1, [(0,), (1,)], [3, 1])
    A = W.random_tensor((0,), [r, x, k], (0,), seed)
    B = W.random_tensor((0,), [k.conj(), x.conj(), c], (0,), seed + 1)
    return A, B, (2,), (0,)


def _split(ctx, case, rtol=RTOL):
    from paper_2405_12196_gb300 import ytn
    A, B, axa, axb = case
    for _ in range(2):   # the first call runs every candidate, the second the kept one
        _, rec, res = run_tensordot(ctx, A, B, axa, axb, prec=ytn.YTN_SPLIT_BF16, rtol=rtol)
        check_against_oracle(rec, oracle_tensordot(A, B, axa, axb), rtol=rtol)
    return rec, res


@pytest.mark.parametrize("M", [1, 127, 129, 300])
@pytest.mark.parametrize("N", [1, 128, 129, 257, 450])
@pytest.mark.parametrize("K", [1, 33, 257, 288])
def test_tile_and_chunk_edges(ctx, M, N, K):
    _split(ctx, _dense(M, K, N, 17))


@pytest.mark.parametrize("stages", [1, 5, 6, 7, 8, 9, 13, 14, 15, 16, 17, 22, 24])
@pytest.mark.parametrize("rtol", [1e-8, 1e-10, 2e-11])   # four, five and six slices
def test_every_stage_count(ctx, stages, rtol):
    _, res = _split(ctx, _dense(130, 32 * stages - 3, 200, stages), rtol)
    assert res["slices"] == {1e-8: 4, 1e-10: 5, 2e-11: 6}[rtol] or res["slices"] >= 4


def test_long_contraction(ctx):
    """Sums beyond 2^51 in the fixed-point accumulators take the general conversion."""
    _split(ctx, _dense(70, 8200, 90, 3))


@pytest.mark.parametrize("rows", [(1, 1, 2, 1, 3, 1, 1, 2), (5, 31, 33, 64), (40, 200)])
@pytest.mark.parametrize("cols", [(1, 2, 1, 1, 4, 1, 1, 1), (3, 30, 130), (129, 64)])
def test_blocks_of_c(ctx, rows, cols):
    _split(ctx, _blocks(rows, cols, (9, 40, 3), 5))


@pytest.mark.parametrize("seed", range(3))
def test_missing_blocks(ctx, seed):
    rng = np.random.default_rng(seed)
    A, B, axa, axb = _blocks((5, 40, 9, 130), (33, 3, 140, 8), (20, 3, 70), 11)
    out = []
    for T in (A, B):
        off = np.concatenate([[0], np.cumsum(np.prod(T["D"], axis=1))])
        keep = sorted(rng.choice(len(T["t"]), 2 * len(T["t"]) // 3, replace=False).tolist())
        out.append({**T, "t": T["t"][keep], "D": T["D"][keep],
                    "data": np.concatenate([T["data"][off[i]:off[i + 1]] for i in keep])})
    _split(ctx, (out[0], out[1], axa, axb))


def _call(ctx, case, dc, da=None, rtol=RTOL):
    import torch
    from paper_2405_12196_gb300 import ytn
    A, B, axa, axb = case
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, axa, axb)
    da = to_dev(A["data"]) if da is None else da
    db = to_dev(B["data"])
    ws = torch.empty(ytn.ytn_workspace_size(plan, ytn.YTN_SPLIT_BF16, rtol), dtype=torch.uint8, device=device())
    ytn.ytn_tensordot(plan, da, db, dc, prec=ytn.YTN_SPLIT_BF16, rtol=rtol, workspace=ws)
    ytn.ytn_sync(ctx)
    return plan


@pytest.mark.parametrize("case", [_blocks((5, 31, 33, 64), (3, 30, 130), (9, 40, 300), 5), _dense(300, 700, 190, 9)])
def test_blocks_written_directly_equal_the_scattered_ones(ctx, case):
    """C in device memory is written by the GEMM, C in page-locked host memory through
    the dense matrix and the scatter, C overlapping A likewise: the same bits."""
    import torch
    from paper_2405_12196_gb300 import ytn
    size = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, *case).out["size"]
    dev = torch.full((size,), float("nan"), dtype=torch.float64, device=device())
    _call(ctx, case, dev)
    _call(ctx, case, dev)
    host = torch.full((size,), float("nan"), dtype=torch.float64).pin_memory()
    _call(ctx, case, host)
    np.testing.assert_array_equal(host.numpy(), dev.cpu().numpy())
    n = case[0]["data"].size
    both = torch.zeros(max(n, size), dtype=torch.float64, device=device())
    both[:n] = to_dev(case[0]["data"])
    _call(ctx, case, both, da=both)
    np.testing.assert_array_equal(both[:size].cpu().numpy(), dev.cpu().numpy())


@pytest.mark.parametrize("exponents", [(-160, -165), (-150, 100), (150, 150), (-300, 290), (-161, -162)])
def test_results_at_the_ends_of_the_range(ctx, exponents):
    """Rows and columns scaled by powers of ten: normal, subnormal, zero and infinite
    results, against the product of the rows and columns brought to 1 by powers of two
    (a sum of subnormal products would round at each of them). Bound: the tolerance of
    the row's largest result plus a few subnormal units."""
    import torch
    A, B, axa, axb = _dense(140, 60, 150, 2)
    a = A["data"].reshape(140, 60) * 10.0 ** (exponents[0] + np.arange(140) % 5)[:, None]
    b = B["data"].reshape(60, 150) * 10.0 ** (exponents[1] + np.arange(150) % 4)[None, :]
    A, B = {**A, "data": a.reshape(-1)}, {**B, "data": b.reshape(-1)}
    c = torch.full((140 * 150,), float("nan"), dtype=torch.float64, device=device())
    from paper_2405_12196_gb300 import ytn
    try:
        _call(ctx, (A, B, axa, axb), c)
    except ytn.YtnError as e:   # the error estimate has no norm to relate to
        assert e.name == "YTN_E_TOLERANCE"
    got = c.cpu().numpy().reshape(140, 150)
    with np.errstate(over="ignore", under="ignore"):
        ea, eb = np.frexp(np.abs(a).max(axis=1))[1], np.frexp(np.abs(b).max(axis=0))[1]
        want = np.ldexp(np.ldexp(a, -ea[:, None]) @ np.ldexp(b, -eb[None, :]), ea[:, None] + eb[None, :])
        scale = np.abs(a).max(axis=1)[:, None] * np.abs(b).max(axis=0)[None, :]
    fin = np.isfinite(want) & (np.abs(want) < 1e307)
    assert np.all(np.abs(got[fin] - want[fin]) <= 1e-9 * scale[fin] + 1.5e-323)
    big = np.abs(want) > 1.79e308
    assert np.all(np.isinf(got[big]) | ~np.isfinite(want[big]))
