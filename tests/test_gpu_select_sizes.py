"""Calls smaller than their context, in a process that has created no other context: the selection keeps the choices in shared
memory up to 8192 of them, so a call of that many needs more of it than one of more rows."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys
import torch
from paper_2602_08404_b200 import binding as B
E, k, ns, G, T = map(int, sys.argv[1:])
H, I = 128, 64
g = torch.Generator(device="cuda").manual_seed(T)
wr, wg, wu, wd, x = (torch.randn(s, generator=g, device="cuda") * 0.1 for s in ((E, H), (E + ns, I, H), (E + ns, I, H), (E + ns, H, I), (T, H)))
wg, wu, wd, x = (v.to(torch.bfloat16) for v in (wg, wu, wd, x))
cfg = B.make_config(H, E, k, I, ns, max_rows=2048, max_groups=G, flags=3)
ctx = B.team_create(cfg)
tiles = B.team_pack_w_tiles(wg, wu, wd)
B.team_set_weights(ctx, wr, w_gu_tiles=tiles[0], w_down_tiles=tiles[1])
t = torch.arange(T, dtype=torch.int32, device="cuda")
st = dict(tok_state=torch.ones(T, dtype=torch.uint8, device="cuda"), conf=torch.ones(T, device="cuda"), pos=t % 16, group=t // 16 % G,
          branch=t // (16 * G))
y, out = [torch.zeros((T, H), device="cuda") for _ in range(2)], B.alloc_routing(cfg, T)
B.team_moe_forward(ctx, x, st, None, y[0])
B.team_moe_forward(ctx, x, st, out, y[1])
assert B.team_read_status(ctx) == (B.TEAM_OK, 0)
own = (x.float() @ wr.T).topk(k, dim=1).indices.sort(dim=1).values
assert (out["topk_idx"].sort(dim=1).values == own).float().mean() > 0.999        # near-ties of the fp32 product
assert int(out["n_rows_active"]) == T and int(out["expert_offset"][-1]) == T * (k + ns)
assert float((y[0] - y[1]).norm() / y[1].norm()) < 1e-5
"""


@pytest.mark.parametrize("E,k,ns,G,T", [(128, 8, 0, 64, 1000), (96, 6, 1, 64, 1200), (128, 8, 0, 1, 1024)])
def test_first_context_of_a_process(E, k, ns, G, T):
    r = subprocess.run([sys.executable, "-c", CODE] + [str(v) for v in (E, k, ns, G, T)], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
