"""The tensor-memory experts work from marks of who chose whom, set where a row is routed (calls without exports) or by a kernel
of its own (calls that export dispatch tables, which are compared with the oracle elsewhere): the outputs of both kinds of call."""
from dataclasses import replace

import pytest
import torch

from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

TOL = 2e-5      # as in test_gpu_inline_select.py: orders of the fp32 sums

S = W.Shape("marks", 256, 24, 4, 192, 0, "bf16", 16, 4, 1, 1, 2, 0.7, seed=41)
CASES = {
    # one row; words of 32 rows; an expert's 128 token-slots exactly, one more, and three chunks; one weight tile per expert
    "1_row": replace(S, block=1),
    "33_rows": replace(S, block=11, seqs=3, n_experts=256, top_k=16, inter=64),
    "128_rows_shared": replace(S, block=32, branches=4, n_shared=1),
    "129_rows_shared": replace(S, block=1, seqs=129, n_shared=4, inter=64),
    "300_rows_of_2_experts": replace(S, block=10, seqs=30, n_experts=2, top_k=2, hidden=384),
    # more pairs of chunks than tiles, every row on every expert; one word more than a warp has lanes, the last with one row
    "2048_rows_of_2_experts": replace(S, block=32, seqs=64, n_experts=2, top_k=2, inter=128, hidden=128),
    "1025_rows_shared": replace(S, block=41, seqs=25, n_experts=12, top_k=5, n_shared=1, inter=64, hidden=128),
    "2048_rows": replace(S, block=32, seqs=64, n_experts=9, top_k=3, inter=64, hidden=128),
}


@pytest.mark.parametrize("flags", [0, 3])
@pytest.mark.parametrize("name", list(CASES))
def test_calls_with_and_without_tables(name, flags):
    shape = CASES[name]
    layer = P.Layer(shape, W.make_weights(shape), flags)
    try:
        for step in W.make_schedule(shape)[:3]:
            x, st = B.to_device(step["x"], B.TEAM_DTYPE_BF16), B.state_to_device(step)
            y, launches = [torch.full((shape.rows, shape.hidden), 7.0, device="cuda") for _ in range(2)], []
            for i, out in enumerate((B.alloc_routing(layer.cfg, shape.rows), None)):
                B.team_moe_forward(layer.ctx, x, st, out, y[i])
                launches.append(B.team_last_launch_count(layer.ctx))
            assert B.team_read_status(layer.ctx)[0] == B.TEAM_OK
            assert launches[1] == 4 < launches[0]
            assert ((y[1] - y[0]).abs() <= TOL * y[0].abs().max(dim=1, keepdim=True).values).all()
            assert torch.equal(y[0] == 7.0, y[1] == 7.0)
    finally:
        layer.close()
