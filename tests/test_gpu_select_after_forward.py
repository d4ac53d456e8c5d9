"""team_select_experts on the logits that a call of team_moe_forward left: the tables that this call exports."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

SHAPES = [W.C1, replace(W.C1, name="c1_9_rows", block=9), replace(W.MINI_BF16, hidden=1024), replace(W.MINI_BF16, hidden=1024, block=31), W.MINI_SHARED]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s.dtype}_{s.rows}")
def test_tables_of_the_last_call(shape):
    layer = P.Layer(shape, W.make_weights(shape), 3)
    try:
        y = torch.zeros((shape.rows, shape.hidden), device="cuda")
        for step in W.make_schedule(shape)[:2]:
            x, st = B.to_device(step["x"], P.dtype_code(shape)), B.state_to_device(step)
            want, got = (B.alloc_routing(layer.cfg, shape.rows) for _ in range(2))
            B.team_moe_forward(layer.ctx, x, st, want, y)
            B.team_route(layer.ctx, -x, st, B.alloc_routing(layer.cfg, shape.rows))        # other logits
            B.team_moe_forward(layer.ctx, x, st, None, y)
            B.team_select_experts(layer.ctx, st, got)
            assert B.team_read_status(layer.ctx)[0] == B.TEAM_OK
            want, got = B.routing_to_host(want), B.routing_to_host(got)
            for n in ("topk_idx", "tok_class", "group_mask", "expert_count", "perm", "active"):
                np.testing.assert_array_equal(got[n], want[n], err_msg=n)
    finally:
        layer.close()
