"""Complex products at the edges of the scatter-combine kernel's chunks (1024 elements
of one output block) against the oracle, for every presence of the quadrants."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import FP64_RTOL, check_against_oracle, device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_12196_gb300 import ytn
    return ytn.ytn_ctx_create(0)


@pytest.mark.parametrize("rows,cols", [((1, 1), (1, 1)), ((1024, 1), (1, 3)), ((1, 31), (33, 1)), ((205, 3), (5, 41)),
                                       ((1, 2), (1025, 4097)), ((64, 17), (48, 129))])
@pytest.mark.parametrize("dts", [("c128", "c128"), ("c128", "f64"), ("f64", "c128")])
def test_complex_scatter_chunks(ctx, rows, cols, dts):
    import torch
    from paper_2405_12196_gb300 import ytn
    t = [(0,), (1,)]
    k = W.Leg(-1, t, [2, 5])
    A = W.random_tensor((0,), [W.Leg(1, t, rows), k], (0,), 3, dtype=dts[0])
    B = W.random_tensor((0,), [k.conj(), W.Leg(-1, t, cols)], (0,), 4, dtype=dts[1])
    plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, A, B, (1,), (0,))
    dev = [torch.from_numpy(np.ascontiguousarray(x["data"])).to(device()) for x in (A, B)]
    c = torch.full((plan.out["size"],), float("nan"), dtype=torch.complex128, device=device())
    ws = torch.empty(ytn.ytn_workspace_size(plan), dtype=torch.uint8, device=device())
    ytn.ytn_tensordot(plan, dev[0], dev[1], c, workspace=ws)
    ytn.ytn_sync(ctx)
    want = O.to_record(O.tensordot(O.from_record(A), O.from_record(B), (1,), (0,)))
    check_against_oracle({**plan.out, "data": c.cpu().numpy()}, want, rtol=FP64_RTOL)
