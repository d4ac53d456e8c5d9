"""Tensor-memory experts: how the work is cut where one expert has many more token-slots than the others (a shared expert), at
the sizes where its cost changes: 32 and 33 slots, a full chunk, one more; odd and even numbers of weight tiles, more CTAs than
steps and fewer.  Every unit of work is done once: outputs against the oracle."""
from dataclasses import replace

import pytest

from paper_2602_08404_b200 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu

S = W.Shape("shared", 256, 64, 2, 128, 1, "bf16", 32, 3, 1, 1, 2, 0.7, seed=63)
CASES = {
    "32_rows": replace(S),
    "33_rows": replace(S, block=33, inter=192),
    "100_rows_wide": replace(S, block=20, seqs=5, hidden=384, n_experts=250, top_k=4, inter=192, n_shared=2),
    "128_rows": replace(S, branches=4, inter=512),
    "129_rows": replace(S, block=43, seqs=3, hidden=640, inter=320),
    # as many rows as a warp lists at once, of an expert with several chunks among small ones
    "1024_rows": replace(S, seqs=32, n_experts=100, hidden=128, inter=64),
    # nobody has four times the mean
    "128_rows_of_3_experts": replace(S, branches=4, n_experts=3, top_k=1, n_shared=2),
}


@pytest.mark.parametrize("flags", [0, 3])
@pytest.mark.parametrize("name", list(CASES))
def test_outputs_with_a_shared_expert(name, flags):
    shape = CASES[name]
    P.run_schedule(shape, W.make_weights(shape), W.make_schedule(shape)[:3], flags, tables=False)
