"""Calls that ask for no table take paths of their own (the one-cluster fp32 step, the selection inside the weight-streaming kernel,
marks set where a row is routed for the tensor-memory kernels): their outputs against the oracle, and with rows that are not
finite among them."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import team_oracle as O
from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

F32 = W.Shape("f32", 256, 16, 2, 128, 0, "f32", 4, 4, 1, 1, 1, 0.7, seed=51)
STREAM = W.Shape("stream", 1024, 40, 4, 64, 0, "bf16", 31, 4, 2, 1, 2, 0.7, seed=52)
TILE = W.Shape("tile", 256, 24, 4, 192, 0, "bf16", 32, 4, 4, 1, 3, 0.7, seed=53)
CASES = {       # shape, launches
    "one_cluster_4_rows": (F32, 1),
    "one_cluster_8_rows_shared": (replace(F32, branches=2, n_experts=33, top_k=5, hidden=384, inter=16, n_shared=2), 1),
    "inline_31_rows": (STREAM, 2),
    "inline_88_rows_of_4_groups_shared": (replace(STREAM, block=11, seqs=4, branches=2, n_experts=129, n_shared=1), 2),
    "marks_128_rows_shared": (replace(TILE, branches=4, n_shared=1, seed=55), 4),
    "marks_320_rows_of_3_experts": (replace(TILE, block=8, seqs=10, branches=4, n_experts=3, top_k=2), 4),
}
# orders of the fp32 sums, as in test_gpu_inline_select.py: the rows that stay finite are computed as before
TOL = 2e-5


@pytest.mark.parametrize("flags", [0, 3])
@pytest.mark.parametrize("name", list(CASES))
def test_outputs_and_rows_that_are_not_finite(name, flags):
    shape, launches = CASES[name]
    weights, ocfg = W.make_weights(shape), P.oracle_config(shape, flags)
    layer = P.Layer(shape, weights, flags)
    try:
        for si, step in enumerate(W.make_schedule(shape)[:3]):
            x, st = B.to_device(step["x"], P.dtype_code(shape)), B.state_to_device(step)
            before = np.full((shape.rows, shape.hidden), 7.0, dtype=np.float32)

            def forward(v, out):
                y = torch.as_tensor(before).cuda()
                B.team_moe_forward(layer.ctx, v, st, out, y)
                assert B.team_last_launch_count(layer.ctx) == launches or out is not None
                return y.cpu().numpy(), B.team_read_status(layer.ctx)

            out = B.alloc_routing(layer.cfg, shape.rows)
            assert forward(x, out)[1] == (B.TEAM_OK, 0)
            (y, status), got = forward(x, None), B.routing_to_host(out)
            assert status == (B.TEAM_OK, 0)
            what = f"{name} flags={flags} step={si}"
            y_ref, ref = O.moe_forward(ocfg, weights, step["x"], step["tok_state"], step["conf"], step["pos"], step["group"], step["branch"],
                                       y_prev=before.astype(np.float64))
            _, pin = P.compare_routing(ocfg, ref, got, step["group"], what, return_pin=True)
            P.compare_y_rows(shape, ocfg, weights, step["x"], y_ref, ref, got, y, pin, before, what)
            # under delayed caching what a cached row's x holds is not used; with plain top-k a row concerns nobody else
            cached = np.flatnonzero(ref["tok_class"] == O.CLS_SKIP)
            rows = cached if flags else np.array([0, shape.rows - 1])
            bad = x.clone()
            bad[rows[::2]], bad[rows[1::2], 3] = float("nan"), float("inf")
            y_bad, status = forward(bad, None)
            assert status == forward(bad, out)[1]          # a row with fewer than k logits above -inf is reported
            rest = np.setdiff1d(np.arange(shape.rows), [] if flags else rows)
            assert (np.abs(y_bad[rest] - y[rest]) <= TOL * np.abs(y[rest]).max(axis=1, keepdims=True)).all(), what
            if not flags:
                assert np.isnan(y_bad[0]).all() and not np.isfinite(y_bad[-1]).all(), what
    finally:
        layer.close()
