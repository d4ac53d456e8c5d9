"""The tensor-memory experts without a dispatch table asked for (the dispatch is formed from the rows' choices alone) and
their steps of two accumulators: experts of one, two and more chunks of 128 token-slots, odd numbers of weight tiles, hardly
any work at all."""
import dataclasses

import pytest

from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

TILE = ((B.TEAM_KNOB_EXPERT_KERNEL, 2),)
# 300 rows on 6 experts: about 150 slots per expert (two chunks) and 300 for the shared one (three); 3 weight tiles of 64
# intermediate columns, 3 of 128 hidden rows
CHUNKS = W.Shape("tile_chunks_bf16", 384, 6, 3, 192, 1, "bf16", 25, 3, 5, 1, 2, 0.7, seqs=12, seed=21)
# as many rows as a chunk holds, and one more, all on all experts
FULL = W.Shape("tile_full_bf16", 256, 2, 2, 64, 0, "bf16", 32, 2, 4, 1, 3, 0.7, seqs=4, seed=22)
OVER = dataclasses.replace(FULL, name="tile_over_bf16", block=43, seqs=3, seed=23)
ONE = W.Shape("tile_one_row_bf16", 128, 200, 4, 64, 0, "bf16", 1, 1, 1, 1, 1, 0.7, seed=24)
# a second batch of choices per row, several shared experts, experts of several warps
TOP12 = W.Shape("tile_top12_bf16", 128, 250, 12, 64, 4, "bf16", 10, 2, 3, 1, 2, 0.7, seqs=7, seed=27)
# more rows than one pass of a CTA's warps takes, in one and in many groups
ROWS = W.Shape("tile_1088_rows_bf16", 128, 40, 3, 64, 2, "bf16", 64, 2, 8, 1, 3, 0.7, seqs=17, seed=25)
WIDE = W.Shape("tile_1100_rows_bf16", 128, 33, 9, 64, 1, "bf16", 11, 2, 3, 1, 3, 0.7, seqs=25, branches=4, seed=31)


@pytest.mark.parametrize("flags", [0, B.TEAM_F_DCD | B.TEAM_F_LAC], ids=["vanilla", "team"])
@pytest.mark.parametrize("shape", [CHUNKS, FULL, OVER, ONE, TOP12, ROWS, WIDE, W.MINI_SHARED, W.MINI_WRAP], ids=lambda s: s.name)
def test_chunks_and_tiles(shape, flags):
    weights = W.make_weights(shape)
    steps = W.make_schedule(shape)
    stats = P.run_schedule(shape, weights, steps, flags, tables=False, knobs=TILE)
    # router, routing rounds, dispatch, two passes
    assert all(s["launches"] == 5 for s in stats)
    stats = P.run_schedule(shape, weights, steps[:1], flags, knobs=TILE)
    assert stats[0]["launches"] >= 5
