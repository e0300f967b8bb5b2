"""Traces with few terms per output element (a thread per element) at the edges of the
kernel's chunks and of the rule that picks it, against the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_against_oracle, device, run_move, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


def _check(ctx, A, ax1, ax2):
    import torch
    from paper_2405_12196_gb300 import ytn
    want = O.to_record(O.trace(O.from_record(A), ax1, ax2))
    if A.get("dtype", "f64") == "f64":
        _, got = run_move(ctx, ytn.YTN_OP_TRACE, A, axa=ax1, axb=ax2)
    else:
        plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TRACE, A, axa=ax1, axb=ax2)
        out = torch.full((2 * plan.out["size"],), float("nan"), dtype=torch.float64, device=device())
        ytn.ytn_trace(plan, to_dev(A["data"].view(np.float64)), out)
        ytn.ytn_sync(ctx)
        got = {**plan.out, "data": out.cpu().numpy().view(np.complex128)}
    check_against_oracle(got, want)


# 16 and 32 terms are the line's ends (17 and 33 beyond it); 127 to 129 elements a CTA's
@pytest.mark.parametrize("diag", [(1,), (1, 1, 2), (16,), (9, 8), (20, 12), (33,)])
@pytest.mark.parametrize("free", [(1, 1), (127, 1), (16, 8), (43, 3), (25, 41)])
@pytest.mark.parametrize("dtype", ["f64", "c128"])
def test_chunk_and_term_edges(ctx, diag, free, dtype):
    d = W.Leg(1, [(q,) for q in range(len(diag))], diag)
    f = [W.Leg(1, [(0,), (1,)], [x, 2]) for x in free]
    A = W.random_tensor((0,), [f[0], d, f[1].conj(), d.conj()], (0,), 3, dtype=dtype)
    _check(ctx, A, (1,), (3,))


@pytest.mark.parametrize("terms", [16, 24, 33])
def test_outputs_beyond_the_line(ctx, terms):
    """55,000 output elements: more than four times what the other kernel holds at once."""
    d, f = W.Leg(1, [(0,)], [terms]), W.Leg(1, [(q,) for q in range(-2, 3)], [54] * 5)
    g = W.Leg(1, [(q,) for q in range(-1, 2)], [70] * 3)
    _check(ctx, W.random_tensor((0,), [d, f, g.conj(), d.conj()], (0,), 4), (0,), (3,))


def test_outputs_of_both_kernels(ctx):
    """Output blocks with one contribution and with all of them: each goes its own way."""
    d = W.Leg(1, [(q,) for q in range(3)], [5, 30, 9])
    f = W.Leg(1, [(q,) for q in range(3)], [11, 40, 7])
    A = W.random_tensor((0,), [d, f, f.conj(), d.conj()], (0,), 5)
    off = np.concatenate([[0], np.cumsum(np.prod(A["D"], axis=1))])
    t = A["t"].reshape(len(A["t"]), -1)
    keep = [i for i in range(len(t)) if t[i][1] == 1 or t[i][0] != 1]   # charge 1 of d with f's charge 1 alone
    A = {**A, "t": A["t"][keep], "D": A["D"][keep], "data": np.concatenate([A["data"][off[i]:off[i + 1]] for i in keep])}
    _check(ctx, A, (0,), (3,))


def test_two_pairs(ctx):
    d, e = W.Leg(1, [(0,), (1,)], [2, 1]), W.Leg(1, [(0,), (1,)], [1, 3])
    f = W.Leg(1, [(0,), (1,)], [30, 9])
    A = W.random_tensor((0,), [d, f, e, f.conj(), e.conj(), d.conj()], (0,), 6)
    _check(ctx, A, (0, 2), (5, 4))
