"""The FP64 grouped GEMM at the edges of its tiles (64, 32, 16 by the plan's size), of
its K steps (1 and 2: multiply-adds; tails of 4 and 16) and of C's blocks, which it
writes itself, against the oracle."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import FP64_RTOL, check_against_oracle, oracle_tensordot, run_tensordot

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _pair(rows, cols, ks, seed=5):
    """A(row legs; k) and B(k; column legs): the row and column dims over three charges
    each, so that C has blocks of several shapes in one sector per charge of k."""
    t = [(q,) for q in range(3)]
    r, c, k = W.Leg(1, t, rows), W.Leg(-1, t, cols), W.Leg(-1, t[:len(ks)], ks)
    x = W.Leg(1, [(0,), (1,)], [2, 1])
    A = W.random_tensor((0,), [r, x, k], (0,), seed)
    B = W.random_tensor((0,), [k.conj(), x.conj(), c], (0,), seed + 1)
    return A, B, (2,), (0,)


@pytest.mark.parametrize("rows", [(1, 2, 1), (7, 9, 15), (16, 17, 1), (31, 64, 33)])
@pytest.mark.parametrize("cols", [(1, 1, 1), (8, 5, 24), (65, 2, 63)])
@pytest.mark.parametrize("ks", [(1, 2, 3), (4, 5, 16), (17, 33, 1)])
def test_small_sectors(ctx, rows, cols, ks):
    A, B, axa, axb = _pair(rows, cols, ks)
    _, rec, _ = run_tensordot(ctx, A, B, axa, axb)
    check_against_oracle(rec, oracle_tensordot(A, B, axa, axb), rtol=FP64_RTOL)


@pytest.mark.parametrize("m", [300, 811, 1601])
@pytest.mark.parametrize("ks", [(1, 2, 3), (2, 4, 19)])
def test_large_sectors(ctx, m, ks):
    A, B, axa, axb = _pair((m, m // 3, 1), (m - 1, 5, m // 2), ks)
    _, rec, _ = run_tensordot(ctx, A, B, axa, axb)
    check_against_oracle(rec, oracle_tensordot(A, B, axa, axb), rtol=FP64_RTOL)


@pytest.mark.parametrize("seed", range(4))
def test_missing_blocks(ctx, seed):
    """Operands without some of their blocks: pairs of row and column blocks that share
    no contracted charge have no block in C and are not written."""
    rng = np.random.default_rng(seed)
    A, B, axa, axb = _pair((5, 40, 9), (33, 3, 8), (2, 3, 70))
    out = []
    for T in (A, B):
        off = np.concatenate([[0], np.cumsum(np.prod(T["D"], axis=1))])
        keep = sorted(rng.choice(len(T["t"]), max(1, len(T["t"]) // 2), replace=False).tolist())
        out.append({**T, "t": T["t"][keep], "D": T["D"][keep],
                    "data": np.concatenate([T["data"][off[i]:off[i + 1]] for i in keep])})
    _, rec, _ = run_tensordot(ctx, out[0], out[1], axa, axb)
    want = oracle_tensordot(out[0], out[1], axa, axb)
    if rec["size"]:
        check_against_oracle(rec, want, rtol=FP64_RTOL)
    else:
        assert np.asarray(want["data"]).size == 0
