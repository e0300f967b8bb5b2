"""Traces at the edges of the trace kernel's work split (32 output elements per CTA,
the terms shared out over the threads that a smaller block leaves free) and scalar
products over merged runs, against the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import check_against_oracle, run_move, to_dev, device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


# (dims of the traced leg, dims of the two free legs): output blocks of 1, 3, 31..33
# and 1025 elements; one term, fewer terms than threads, many terms
@pytest.mark.parametrize("diag,free", [((1,), (1, 1)), ((5, 1), (3, 1)), ((700, 300), (1, 1)), ((2, 3, 1), (31, 1)),
                                       ((40, 7), (8, 4)), ((3,), (11, 3)), ((9, 130), (41, 25))])
@pytest.mark.parametrize("pairs", [1, 2])
@pytest.mark.parametrize("dtype", ["f64", "c128"])
def test_trace_chunk_edges(ctx, diag, free, pairs, dtype):
    from paper_2405_12196_gb300 import ytn
    if pairs == 2 and max(diag) > 40:
        diag = tuple(min(d, 40) for d in diag)
    t = [(q,) for q in range(len(diag))]
    d, f = W.Leg(1, t, diag), [W.Leg(1, [(0,)], [x]) for x in free]
    legs = [d, f[0], f[1].conj(), d.conj()]
    ax1, ax2 = (0,), (3,)
    if pairs == 2:
        e = W.Leg(1, [(0,), (1,)], [2, 3])
        legs = [d, e, f[0], e.conj(), f[1].conj(), d.conj()]
        ax1, ax2 = (0, 1), (5, 3)
    A = W.random_tensor((0,), legs, (0,), 7, dtype=dtype)
    want = O.to_record(O.trace(O.from_record(A), ax1, ax2))
    if dtype == "f64":
        _, got = run_move(ctx, ytn.YTN_OP_TRACE, A, axa=ax1, axb=ax2)
        check_against_oracle(got, want)
        return
    import torch
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TRACE, A, axa=ax1, axb=ax2)
    out = torch.full((2 * plan.out["size"],), float("nan"), dtype=torch.float64, device=device())
    ytn.ytn_trace(plan, to_dev(A["data"].view(np.float64)), out)
    ytn.ytn_sync(ctx)
    check_against_oracle({**plan.out, "data": out.cpu().numpy().view(np.complex128)}, want)


@pytest.mark.parametrize("sizes", [[4095, 1, 1, 4096, 4097, 3], [1] * 70, [8192, 5, 12289]])
@pytest.mark.parametrize("drop", [(), (1,), (0, 3)])
def test_vdot_runs_over_block_boundaries(ctx, sizes, drop):
    """Runs that join blocks end where one tensor lacks a block, at 4096 elements and at
    a CTA's share; bound: 1e-13 of the sum of the magnitudes."""
    import torch
    from paper_2405_12196_gb300 import ytn
    legs = [W.Leg(1, [(q,) for q in range(len(sizes))], sizes),
            W.Leg(-1, [(q,) for q in range(len(sizes))], [1] * len(sizes))]
    A, B = W.random_tensor((0,), legs, (0,), 1), W.random_tensor((0,), legs, (0,), 2)
    keep = [i for i in range(len(sizes)) if i not in drop]
    off = np.concatenate([[0], np.cumsum(sizes)])
    B = {**B, "t": B["t"][keep], "D": B["D"][keep],
         "data": np.concatenate([B["data"][off[i]:off[i + 1]] for i in keep])}
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_VDOT, A, B)
    out = torch.empty(1, dtype=torch.float64, device=device())
    ws = torch.empty(max(ytn.ytn_workspace_size(plan), 256), dtype=torch.uint8, device=device())
    ytn.ytn_vdot(plan, to_dev(A["data"]), to_dev(B["data"]), out, workspace=ws)
    ytn.ytn_sync(ctx)
    common = np.concatenate([A["data"][off[i]:off[i + 1]] for i in keep])
    assert abs(out.item() - O.vdot(O.from_record(A), O.from_record(B))) <= 1e-13 * np.abs(common * B["data"]).sum()
