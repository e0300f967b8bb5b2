"""The split GEMM with four and six slices (rings of their own) at the edges of its tiles,
stages and blocks; the slice count is part of the check."""
import pytest

import workloads as W
from gpu_helpers import check_against_oracle, oracle_tensordot, run_tensordot

pytestmark = pytest.mark.gpu

# the smallest s with 128 (2^(-8 s - 1) + 2^-43) <= rtol
SLICES = {2e-8: 4, 1e-8: 5, 6e-11: 6, 2e-11: 6}


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _dense(M, K, N, seed):
    t = [(0,)]
    A = W.random_tensor((0,), [W.Leg(1, t, [M]), W.Leg(-1, t, [K])], (0,), seed)
    B = W.random_tensor((0,), [W.Leg(1, t, [K]), W.Leg(-1, t, [N])], (0,), seed + 1)
    return A, B, (1,), (0,)


def _blocks(rows, cols, ks, seed):
    r = W.Leg(1, [(q,) for q in range(len(rows))], rows)
    c = W.Leg(-1, [(q,) for q in range(len(cols))], cols)
    k = W.Leg(-1, [(q,) for q in range(len(ks))], ks)
    x = W.Leg(1, [(0,), (1,)], [3, 1])
    A = W.random_tensor((0,), [r, x, k], (0,), seed)
    B = W.random_tensor((0,), [k.conj(), x.conj(), c], (0,), seed + 1)
    return A, B, (2,), (0,)


def _split(ctx, case, rtol):
    from paper_2405_12196_gb300 import ytn
    A, B, axa, axb = case
    want = oracle_tensordot(A, B, axa, axb)
    for _ in range(2):   # the first call runs every candidate, the second the kept one
        _, rec, res = run_tensordot(ctx, A, B, axa, axb, prec=ytn.YTN_SPLIT_BF16, rtol=rtol)
        assert res["slices"] == SLICES[rtol]
        if len(rec["t"]) == 1 and rec["size"] >= 1000:   # (a small sector may cancel and be recomputed)
            assert res["report"]["nfallback"] == 0
        check_against_oracle(rec, want, rtol=rtol)


@pytest.mark.parametrize("rtol", [2e-8, 1e-8, 6e-11])
def test_slice_counts(ctx, rtol):
    _split(ctx, _dense(40, 30, 50, 1), rtol)


@pytest.mark.parametrize("rtol", [2e-8, 2e-11])
@pytest.mark.parametrize("M,N", [(1, 1), (127, 129), (129, 60), (300, 257), (130, 450), (257, 190)])
@pytest.mark.parametrize("K", [1, 33, 257, 545])
def test_tile_edges(ctx, M, N, K, rtol):
    _split(ctx, _dense(M, K, N, 17), rtol)


@pytest.mark.parametrize("rtol", [2e-8, 2e-11])
@pytest.mark.parametrize("stages", [1, 2, 3, 4, 5, 7, 8, 9, 14, 16, 17, 24])
def test_stage_counts(ctx, stages, rtol):
    _split(ctx, _dense(300, 32 * stages - 3, 200, stages), rtol)


@pytest.mark.parametrize("rtol", [2e-8, 2e-11])
@pytest.mark.parametrize("rows", [(1, 1, 2, 1, 3, 1, 1, 2), (5, 31, 33, 64), (40, 200)])
@pytest.mark.parametrize("cols", [(1, 2, 1, 1, 4, 1, 1, 1), (3, 30, 130), (129, 64)])
def test_blocks_of_c(ctx, rows, cols, rtol):
    _split(ctx, _blocks(rows, cols, (9, 40, 3), 5), rtol)
