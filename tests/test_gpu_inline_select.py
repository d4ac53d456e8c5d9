"""Calls of few rows that ask for no routing tables are routed inside the expert kernel: their outputs against those of
the same call with every table exported, which goes through the selection kernel and is compared with the oracle elsewhere.
Same choices, same weights, other orders of the fp32 sums."""
from dataclasses import replace

import pytest
import torch

from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

# an output is a sum of at most 20 experts' contributions, each added in at most 64 parts: 1280 roundings of 2^-24, walking
# randomly (36 of them) over partial sums a few times as large as the result; another choice or weight shows at 1e-3
TOL = 2e-5

S1 = W.Shape("stream", 1024, 40, 4, 64, 0, "bf16", 11, 4, 1, 1, 1, 0.7, seed=31)
CASES = {
    # both row tiles, words of 32 rows, experts with several items, more experts than one warp scans
    "9_rows": replace(S1, block=9, n_shared=2),
    "31_rows": replace(S1, block=31, hidden=2048, n_experts=256, top_k=16),
    "33_rows_of_3_groups": replace(S1, seqs=3, n_experts=7, top_k=5),
    "64_rows_one_group": replace(S1, block=64, n_experts=129, inter=192, n_shared=4),
    "65_rows_of_13_groups": replace(S1, seqs=13, block=5, hidden=2048),
    "95_rows": replace(S1, seqs=5, block=19, n_experts=16, top_k=7, L_hot=2),
}


def _both(ctx, cfg, shape, x, st):
    """(outputs, x after the residual add, launches) with every table exported and with none."""
    y = [torch.full((shape.rows, shape.hidden), 7.0, device="cuda") for _ in range(2)]
    add, launches = [x.clone() for _ in range(2)], []
    for i, out in enumerate((B.alloc_routing(cfg, shape.rows), None)):
        B.team_moe_forward(ctx, x, st, out, y[i])
        launches.append(B.team_last_launch_count(ctx))
        B.team_residual_add(ctx, add[i], y[i], shape.rows)       # reads the classes that the call left
    assert B.team_read_status(ctx)[0] == B.TEAM_OK
    return y, add, launches


@pytest.mark.parametrize("flags", [0, 1, 2, 3])
@pytest.mark.parametrize("name", list(CASES))
def test_outputs_without_tables(name, flags):
    shape = CASES[name]
    weights = W.make_weights(shape)
    kw = dict(norm_topk=0) if flags == 1 else {}
    for max_groups in {shape.seqs, 64 if flags == 3 else shape.seqs}:      # more groups than the call has, too
        layer = P.Layer(replace(shape, seqs=max_groups), weights, flags, max_rows=shape.rows, **kw)
        try:
            for step in W.make_schedule(shape)[:3]:
                y, add, launches = _both(layer.ctx, layer.cfg, shape, B.to_device(step["x"], B.TEAM_DTYPE_BF16), B.state_to_device(step))
                assert launches[1] == 2 < launches[0], launches
                assert ((y[1] - y[0]).abs() <= TOL * y[0].abs().max(dim=1, keepdim=True).values).all()
                assert torch.equal(y[0] == 7.0, y[1] == 7.0)
                assert (add[0] != add[1]).float().mean() < 1e-3        # a bf16 rounding that the fp32 difference turns
        finally:
            layer.close()


def test_group_out_of_range_is_reported():
    shape = CASES["33_rows_of_3_groups"]
    layer = P.Layer(shape, W.make_weights(shape), 3)
    try:
        step = W.make_schedule(shape)[1]
        step["group"] = step["group"].copy()
        step["group"][-1] = shape.seqs
        B.team_moe_forward(layer.ctx, B.to_device(step["x"], B.TEAM_DTYPE_BF16), B.state_to_device(step), None,
                           torch.zeros((shape.rows, shape.hidden), device="cuda"))
        assert B.team_read_status(layer.ctx) == (B.TEAM_ERR_STATE, 1)
    finally:
        layer.close()


@pytest.mark.parametrize("rank", [0, 1])
def test_expert_parallel_rank_without_tables(rank):
    from tests.test_gpu_ep import _rank_layer
    shape = replace(S1, seqs=5)
    step = W.make_schedule(shape)[1]
    ctx, cfg, _ = _rank_layer(shape, W.make_weights(shape), 3, rank, 2)
    try:
        y, _, _ = _both(ctx, cfg, shape, B.to_device(step["x"], B.TEAM_DTYPE_BF16), B.state_to_device(step))
        assert ((y[1] - y[0]).abs() <= TOL * y[0].abs().max(dim=1, keepdim=True).values).all()
    finally:
        B.team_destroy(ctx)


F1 = W.Shape("f32", 256, 16, 2, 128, 0, "f32", 4, 4, 1, 1, 1, 0.7, seed=33)
F32_CASES = {
    "1_row": replace(F1, block=1, n_experts=1, top_k=1),
    "8_rows_of_2_branches": replace(F1, branches=2, n_experts=31, top_k=5, hidden=252, inter=32, n_shared=2),
    "8_rows_of_8_groups": replace(F1, block=1, seqs=8, n_experts=256, top_k=16, hidden=64, inter=16),
    "hidden_4100": replace(F1, block=3, hidden=4100, inter=16, top_k=1),
    "most_weights": replace(F1, block=4, hidden=512, inter=80, top_k=2),
    "too_many_weights": replace(F1, block=4, hidden=512, inter=96, top_k=2),
    "9_rows": replace(F1, block=9),
}


@pytest.mark.parametrize("flags", [0, 3])
@pytest.mark.parametrize("name", list(F32_CASES))
def test_fp32_step_without_tables(name, flags):
    """The one-cluster step of fp32 configurations against the four kernels, which sum the logits and the down product in
    another order: 1e-5 covers what a logit's rounding (2e-7 of values below 5) does to the routing weights, and sums of at
    most 256 terms (16 roundings of 2^-24 on a random walk).  The down product's 2, 4 and 8 columns per warp: 1_row and
    8_rows_of_8_groups, 8_rows_of_2_branches and most_weights, hidden_4100 (whose last piece is half empty)."""
    shape = F32_CASES[name]
    layer = P.Layer(shape, W.make_weights(shape), flags, **(dict(norm_topk=0) if flags == 0 else {}))
    try:
        for step in W.make_schedule(shape)[:3]:
            y, add, launches = _both(layer.ctx, layer.cfg, shape, B.to_device(step["x"], B.TEAM_DTYPE_F32), B.state_to_device(step))
            assert launches == ([4, 4] if name in ("too_many_weights", "9_rows") else [4, 1])
            assert ((y[1] - y[0]).abs() <= 1e-5 * y[0].abs().max(dim=1, keepdim=True).values).all()
            assert torch.equal(y[0] == 7.0, y[1] == 7.0)
            assert ((add[1] - add[0]).abs() <= 1e-5 * add[0].abs().max()).all()
    finally:
        layer.close()


@pytest.mark.parametrize("rows,hidden,n_experts,launches", [(4, 4096, 256, 4), (8, 1024, 128, 1), (8, 1024, 129, 4), (1, 2048, 256, 1)])
def test_fp32_step_router_weights(rows, hidden, n_experts, launches):
    """The router's weights count, too: the one-cluster step is for calls whose weights one cluster reads faster."""
    shape = replace(F1, block=rows, hidden=hidden, n_experts=n_experts, top_k=1, inter=16)
    layer = P.Layer(shape, W.make_weights(shape), 0)
    try:
        step = W.make_schedule(shape)[1]
        y, _, got = _both(layer.ctx, layer.cfg, shape, B.to_device(step["x"], B.TEAM_DTYPE_F32), B.state_to_device(step))
        assert got == [4, launches]
        assert ((y[1] - y[0]).abs() <= 1e-5 * y[0].abs().max(dim=1, keepdim=True).values).all()
    finally:
        layer.close()


@pytest.mark.parametrize("rank", [0, 1])
def test_fp32_expert_parallel_rank_without_tables(rank):
    from tests.test_gpu_ep import _rank_layer
    step = W.make_schedule(F1)[1]
    ctx, cfg, _ = _rank_layer(F1, W.make_weights(F1), 3, rank, 2)
    try:
        y, _, _ = _both(ctx, cfg, F1, B.to_device(step["x"], B.TEAM_DTYPE_F32), B.state_to_device(step))
        assert ((y[1] - y[0]).abs() <= 1e-5 * y[0].abs().max(dim=1, keepdim=True).values).all()
    finally:
        B.team_destroy(ctx)


@pytest.mark.parametrize("shape,name", [(F1, "k_step_f32"), (F32_CASES["9_rows"], "k_gate_up"), (CASES["31_rows"], "k_experts_stream (selection"),
                                        (replace(S1, block=8), "k_experts_stream (fused")], ids=["one_cluster", "fp32", "inline", "fused"])
def test_expert_kernel_name(shape, name):
    """The kernel that a call of max_rows rows without tables launches; with the knob the general one."""
    ctx = B.team_create(P.lib_config(shape, 3))
    try:
        assert B.team_expert_kernel_name(ctx).startswith(name)
        B.team_debug_knob(ctx, B.TEAM_KNOB_NO_FUSE, 1)
        assert B.team_expert_kernel_name(ctx) in ("k_gate_up + k_down", "k_experts_stream")
    finally:
        B.team_destroy(ctx)
