"""The calls whose speed is followed: the MoE layer of one denoising step (device and host buffers), the attention
half of delayed caching, and the decode loop of a block, each through its public entry point.

A case is a dict of plain values:

  kind "layer"   team_moe_forward, everything on the device
  kind "host"    team_moe_forward_host: activations and step state in pinned host memory, y back in host memory
  kind "attn"    team_block_attention once for each of `layers` layers, every layer with KV caches of its own
  kind "decode"  the passes of a block: team_seh_step, then team_moe_forward on the rows that it laid out

Layer shapes are the ones of paper_2602_08404_b200.workloads (the configurations that the tests and bench.py run) or
generic; rows are [sequence][branch][position], and a context is created for `max_rows` rows like a server's, which
may be more than a call presents.  Every state has weights of its own (random, N(0, 0.02)), so the experts' weights
come from HBM as they do in a model of many layers.
"""
from dataclasses import replace

import numpy as np
import torch

from paper_2602_08404_b200 import binding as B
from paper_2602_08404_b200 import workloads as W

TEAM = B.TEAM_F_DCD | B.TEAM_F_LAC
SDAR = dict(H=2048, E=128, k=8, I=768, ns=0, dtype="bf16")        # one layer of the headline configuration
LLADA = dict(H=2048, E=256, k=8, I=512, ns=1, dtype="bf16")       # 256 experts and an always-on one
TILE_MIN_ROWS = 96      # from here on (or where hidden is not 1024 or 2048) a context reads the tile-major weights


def listed():
    layer = dict(kind="layer", flags=TEAM, L_hot=3)
    return [
        # the fp32 configuration: launch latency and nothing else
        dict(layer, name="layer_f32_tiny", H=256, E=16, k=2, I=128, ns=0, dtype="f32", seqs=1, branches=1, block=4, step=2,
             L_hot=1, max_rows=4),
        # one sequence, block of 4: the latency-bound decoding step, bench.py's default workload
        dict(layer, name="layer_sdar_4rows", **SDAR, seqs=1, branches=1, block=4, step=2, L_hot=1, max_rows=4),
        # the same step for a caller whose buffers are on the host: bench.py's end-to-end figure
        dict(layer, name="host_sdar_4rows", **SDAR, seqs=1, branches=1, block=4, step=2, L_hot=1, max_rows=4) | dict(kind="host"),
        # one sequence, block of 32, a shared expert
        dict(layer, name="layer_llada_32rows", **LLADA, seqs=1, branches=1, block=32, step=3, max_rows=32),
        # a small batch with speculative branches: four sequences x 4 branches x 4
        dict(layer, name="layer_sdar_64rows", **SDAR, seqs=4, branches=4, block=4, step=2, L_hot=1, max_rows=64),
        # the operating point of the paper's experiments: one sequence, block of 32 x 4 branches
        dict(layer, name="layer_sdar_128rows", **SDAR, seqs=1, branches=4, block=32, step=3, max_rows=128),
        # nothing is a round number: 37 sequences in blocks of 5, presented to a context made for 256 rows
        dict(layer, name="layer_odd_185rows", H=1536, E=96, k=6, I=704, ns=1, dtype="bf16", seqs=37, branches=1, block=5, step=2,
             L_hot=2, max_rows=256),
        # a full batch with speculative branches
        dict(layer, name="layer_sdar_1024rows", **SDAR, seqs=64, branches=4, block=4, step=2, L_hot=1, max_rows=1024),
        # the largest call, plain top-k (the baseline that the activation rule is compared with, and what prefill-like
        # passes over many tokens look like)
        dict(layer, name="layer_sdar_2048rows", **SDAR, seqs=64, branches=1, block=32, step=1, max_rows=2048) | dict(flags=0),
        # attention of one forward pass over 16 layers: one sequence, block of 32 x 4 branches, 4096 cached tokens
        dict(name="attn_d128_p4096", kind="attn", flags=B.TEAM_F_DCD, head_dim=128, n_heads=32, n_kv=4, seqs=1, branches=4, block=32,
             step=3, prefix=4096, layers=16),
        # ... of a small batch without branches, head size 64, prefixes of ragged lengths up to 1500
        dict(name="attn_d64_ragged", kind="attn", flags=B.TEAM_F_DCD, head_dim=64, n_heads=16, n_kv=4, seqs=6, branches=1, block=16,
             step=2, prefix=1500, layers=16),
        # decoding: 8 passes over a block of 32 x 4 branches
        dict(name="decode_block32", kind="decode", **SDAR, flags=TEAM, L_hot=3, seqs=1, block=32, branches=4, passes=8, max_rows=128),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _rows(rng, most):
    """(seqs, branches, block) of at most `most` rows, the rows spread over the logarithm."""
    rows = _log(rng, 1, most)
    branches = rng.choice([1, 1, 4]) if rows >= 4 else 1
    block = min(_log(rng, 1, 64), max(1, rows // branches))
    return min(1024, max(1, rows // (branches * block))), branches, block


def _step(rng, block):
    """A step of the scripted block at which something is still computed."""
    return rng.randint(0, min(4, (block - 1) // max(1, block // 8) + 1))


def _draw_layer(rng, kind):
    if kind == "layer" and rng.random() < 0.1:
        c = dict(H=64 * rng.randint(1, 8), E=rng.randint(8, 32), I=16 * rng.randint(2, 16), ns=0, dtype="f32", k=rng.randint(1, 4))
        most = 64
    else:
        H = rng.choice([1024, 2048, 2048, 128 * rng.randint(2, 16)])
        c = dict(H=H, E=_log(rng, 16, 256), I=64 * rng.randint(1, 16), ns=rng.choice([0, 0, 1]), dtype="bf16", k=rng.randint(2, 8))
        most = 64 if kind == "host" else 2048
    seqs, branches, block = _rows(rng, most)
    rows = seqs * branches * block
    max_rows = rows if rng.random() < 0.5 else min(2048, 1 << (rows - 1).bit_length())
    return dict(kind=kind, **c, seqs=seqs, branches=branches, block=block, step=_step(rng, block), L_hot=rng.randint(1, 3),
                max_rows=max_rows, flags=rng.choice([TEAM, TEAM, B.TEAM_F_DCD, 0]))


def _draw_attn(rng):
    seqs, branches, block = _rows(rng, 512)
    n_kv = rng.choice([1, 2, 4, 8])
    return dict(kind="attn", flags=rng.choice([B.TEAM_F_DCD, B.TEAM_F_DCD, 0]), head_dim=rng.choice([64, 128]), n_heads=n_kv * rng.randint(1, 8),
                n_kv=n_kv, seqs=seqs, branches=branches, block=block, step=_step(rng, block), prefix=_log(rng, 16, 8192),
                layers=rng.choice([4, 8, 16]))


def _draw_decode(rng):
    c = _draw_layer(rng, "decode")
    block = rng.choice([8, 16, 32, 32, 48])
    seqs = _log(rng, 1, 6)
    branches = rng.choice([1, 4])
    c.pop("step")
    return dict(c, block=block, seqs=seqs, branches=branches, passes=rng.randint(2, 8), max_rows=seqs * branches * block)


def draw(rng):
    top = {}
    for c in listed():
        w = work(c)
        for n, v in w.items():
            top[n] = max(top.get(n, 0), v)
    while True:
        p = rng.random()
        c = (_draw_layer(rng, "layer") if p < 0.6 else _draw_layer(rng, "host") if p < 0.7 else
             _draw_attn(rng) if p < 0.9 else _draw_decode(rng))
        w = work(c)
        kv = c["layers"] * c["seqs"] * c["prefix"] * c["n_kv"] * c["head_dim"] * 4 if c["kind"] == "attn" else 0
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"] and kv <= 4 << 30:
            return c


# ---- states -------------------------------------------------------------------------------------------------------
def _shape(c):
    steps = c.get("passes") or c.get("step", 0) + 1
    return W.Shape("case", c.get("H", 16), c.get("E", 0), c.get("k", 0), c.get("I", 0), c.get("ns", 0), c.get("dtype", "bf16"), c["block"],
                   steps, max(1, c["block"] // 8), 1, c.get("L_hot", 1), 0.7, seqs=c["seqs"], branches=c["branches"])


class _Layer:
    """A context and the weights that it borrows."""

    def __init__(self, c, seed):
        sh = _shape(c)
        f32 = c["dtype"] == "f32"
        wr, wg, wu, wd = W.device_layer_weights(sh, seed, "cuda")
        cfg = B.make_config(c["H"], c["E"], c["k"], c["I"], c["ns"], max_rows=c["max_rows"], max_groups=c["seqs"],
                            dtype=B.TEAM_DTYPE_F32 if f32 else B.TEAM_DTYPE_BF16, flags=c["flags"], L_hot=c["L_hot"])
        self.ctx = B.team_create(cfg)
        # the layout that a context of this many rows reads (team.h); the row-major source is dropped
        if f32 or (c["max_rows"] < TILE_MIN_ROWS and c["H"] in (1024, 2048)):
            self.w = [wr, wg, wu, B.team_pack_w_down(wd)]
            B.team_set_weights(self.ctx, *self.w)
        else:
            self.w = [wr, *B.team_pack_w_tiles(wg, wu, wd)]
            B.team_set_weights(self.ctx, wr, w_gu_tiles=self.w[1], w_down_tiles=self.w[2])

    def __del__(self):
        if getattr(self, "ctx", None):
            B.team_destroy(self.ctx)
            self.ctx = None


def _step_host(c, seed):
    """Hidden states and step state of the case's step of a scripted block."""
    return W.make_schedule(_shape(c), seed=seed)[c["step"]]


def prepare(case, seed):
    c = dict(case)
    s = dict(case=c)
    if c["kind"] == "attn":
        sh = _shape(c)
        T, L, S, n, d = sh.rows, c["block"], c["seqs"], c["layers"], c["head_dim"]
        g = torch.Generator(device="cuda").manual_seed(seed)

        def normal(*dims):
            return torch.randn(dims, generator=g, device="cuda", dtype=torch.float32).to(torch.bfloat16)

        s["st"] = B.state_to_device(_step_host(c, seed))
        s["q"], s["k_new"], s["v_new"] = normal(n, T, c["n_heads"], d), normal(n, T, c["n_kv"], d), normal(n, T, c["n_kv"], d)
        s["k_prefix"], s["v_prefix"] = normal(n, S, c["prefix"], c["n_kv"], d), normal(n, S, c["prefix"], c["n_kv"], d)
        s["k_block"], s["v_block"] = normal(n, S, L, c["n_kv"], d), normal(n, S, L, c["n_kv"], d)
        rng = np.random.default_rng(seed)
        plen = rng.integers(c["prefix"] // 2, c["prefix"] + 1, S).astype(np.int32)
        plen[0] = c["prefix"]
        s["prefix_len"] = torch.as_tensor(plen).cuda()
        s["out"] = torch.zeros((n, T, c["n_heads"], d), dtype=torch.float32, device="cuda")
        s["status"] = torch.zeros(2, dtype=torch.int32, device="cuda")
        s["calls"] = [tuple(s[n][i] for n in ("q", "k_new", "v_new", "k_prefix", "v_prefix", "k_block", "v_block", "out")) for i in range(n)]
        s["cfg"] = B.team_attn_config(c["n_heads"], c["n_kv"], d, L, S, c["branches"], c["prefix"], c["flags"])
        return s
    s["layer"] = _Layer(c, seed)
    dc = B.TEAM_DTYPE_F32 if c["dtype"] == "f32" else B.TEAM_DTYPE_BF16
    if c["kind"] == "decode":
        sh = _shape(c)
        s["x"] = [B.to_device(st["x"], dc) for st in W.make_schedule(sh, seed=seed)]
        pred, conf = W.make_decode_script(c["seqs"], c["block"], c["passes"], seed, n_branches=c["branches"])
        s["pred"] = [torch.as_tensor(p).contiguous().cuda() for p in pred]
        s["conf"] = [torch.as_tensor(p).contiguous().cuda() for p in conf]
        s["seh"], s["rows"] = B.seh_alloc(c["seqs"], c["block"], c["branches"])
        s["y"] = torch.zeros((sh.rows, c["H"]), dtype=torch.float32, device="cuda")
        return s
    st = _step_host(c, seed)
    T = st["tok_state"].shape[0]
    if c["kind"] == "host":
        x = torch.as_tensor(st["x"])
        s["x"] = (x if c["dtype"] == "f32" else x.to(torch.bfloat16)).contiguous().pin_memory()
        s["st"] = {n: torch.as_tensor(np.ascontiguousarray(st[n])).pin_memory() for n in ("tok_state", "conf", "pos", "group", "branch")}
        s["y"] = torch.zeros((T, c["H"]), dtype=torch.float32).pin_memory()
        s["stream"] = torch.cuda.Stream()
    else:
        s["x"] = B.to_device(st["x"], dc)
        s["st"] = B.state_to_device(st)
        s["y"] = torch.zeros((T, c["H"]), dtype=torch.float32, device="cuda")
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "layer":
        B.team_moe_forward(s["layer"].ctx, s["x"], s["st"], None, s["y"])
        return s["y"]
    if c["kind"] == "host":
        with torch.cuda.stream(s["stream"]):
            B.team_moe_forward_host(s["layer"].ctx, s["x"], s["st"], None, s["y"])
        return s["y"]
    if c["kind"] == "attn":
        for q, k_new, v_new, k_prefix, v_prefix, k_block, v_block, out in s["calls"]:
            rc = B.team_block_attention(s["cfg"], s["st"], q, k_new, v_new, k_prefix, v_prefix, s["prefix_len"], k_block, v_block, out,
                                        s["status"])
            if rc != B.TEAM_OK:
                raise B.TeamError(f"team error {rc}")
        return s["out"], s["k_block"], s["v_block"]
    # decode: begin the block, then one acceptance step in front of every pass but the first
    B.team_seh_step(c["seqs"], c["block"], c["branches"], 0.95, s["seh"], None, None, s["rows"])
    for p in range(c["passes"]):
        B.team_moe_forward(s["layer"].ctx, s["x"][p], s["rows"], None, s["y"])
        B.team_seh_step(c["seqs"], c["block"], c["branches"], 0.95, s["seh"], s["pred"][p], s["conf"][p], s["rows"])
    return s["y"], s["seh"]["token"], s["seh"]["state"], s["rows"]["tok_state"], s["rows"]["conf"]


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def _active(c, rows):
    """About how many routed experts a call activates.  Sequences choose independently; the rows of one sequence are
    alike, and the limited activation keeps the cold ones inside the set of the others: the exponents are fitted to
    the activated sets that bench.py counts on these workloads."""
    per_seq = 1 - (1 - c["k"] / c["E"]) ** (rows ** (0.55 if c["flags"] & B.TEAM_F_LAC else 0.72))
    return c["E"] * (1 - (1 - per_seq) ** c["seqs"])


def work(case):
    c = dict(case)
    T = c["seqs"] * c["branches"] * c["block"]
    st = [W.base_states(_shape(c), p) for p in (range(c["passes"]) if c["kind"] == "decode" else [c["step"]])]
    out = dict(bytes=0.0, flops=0.0)
    for states in st:
        cached = int((states == W.TOK_CACHED).sum()) if c["flags"] & B.TEAM_F_DCD else 0
        rows = T * (c["block"] - cached) / c["block"]
        if c["kind"] == "attn":
            d, n = c["head_dim"], c["layers"]
            mean_prefix = c["prefix"] * (1 + 0.75 * (c["seqs"] - 1)) / c["seqs"]
            keys = mean_prefix + c["block"]
            out["bytes"] += n * (4 * c["seqs"] * keys * c["n_kv"] * d + rows * (c["n_heads"] * d * 6 + c["n_kv"] * d * 4))
            out["flops"] += n * 4 * rows * c["n_heads"] * keys * d
        else:
            elt = 4 if c["dtype"] == "f32" else 2
            experts = (_active(c, rows / c["seqs"]) if rows else 0) + (c["ns"] if rows else 0)
            out["bytes"] += experts * 3 * c["H"] * c["I"] * elt + 4 * c["E"] * c["H"] + rows * c["H"] * (elt + 4)
            out["flops"] += rows * (6 * c["H"] * c["I"] * (c["k"] + c["ns"]) + 2 * c["H"] * c["E"])
    out["bytes"] += 17 * T
    return out


def tolerance(case):
    """About four times the distance that was seen between the path and the same path in 64 bits on its own choices."""
    if case["kind"] == "attn":
        return {"rel": 2e-5, "max": 2e-4}            # seen: 3.5e-6, 2.7e-5
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}            # 32-bit sums
    # seen: 1.7e-3, 1.3e-2 (the activations are rounded to bf16 once).  Where a call has many rows, the last choice of
    # one of them may be a tie within the rounding of its logits: another expert of the same weight then stands in.
    many = case["seqs"] * case["branches"] * case["block"] >= TILE_MIN_ROWS
    return {"rel": 7e-3, "max": 0.9 if many else 0.06}


# ---- what run returns, in 64 bits -----------------------------------------------------------------------------------
def _classes(c, states, conf):
    """True for rows that are computed, and for those among them that choose in the first round, [S, B, L] each: Eq. 4 with
    make_config's defaults (threshold 0.7, a distance of at most L_hot, the position in front of the block decoded)."""
    S, nb, L = states.shape
    decoded = np.concatenate([np.ones((S, nb, 1), bool), states != W.TOK_MASKED], axis=2)
    near_by = np.abs(np.arange(L)[:, None] - np.arange(-1, L)[None, :]) <= c["L_hot"]
    near = (decoded[:, :, None, :] & near_by).any(axis=3)
    computed = (states != W.TOK_CACHED) | (not c["flags"] & B.TEAM_F_DCD)
    first = computed & ((states != W.TOK_MASKED) | (conf > np.float32(0.7)) | near | (not c["flags"] & B.TEAM_F_LAC))
    empty = ~first.any(axis=(1, 2))
    first[empty] = computed[empty]
    return computed, first


def _layer64(c, weights, x, states, conf, y):
    """The layer on x [T, H]; rows that are not computed keep what y holds.  Experts are chosen on the 64-bit logits."""
    wr, wg, wu, wd = weights
    computed, first = _classes(c, states.reshape(c["seqs"], -1, c["block"]), conf.reshape(c["seqs"], -1, c["block"]))
    S, T = c["seqs"], x.shape[0]
    computed, first = (torch.as_tensor(a.reshape(S, -1)).cuda() for a in (computed, first))
    x64 = x.double()
    logits = x64 @ wr.double().T
    own = torch.zeros(logits.shape, dtype=torch.bool, device="cuda").scatter_(1, logits.topk(c["k"], dim=1).indices, True).view(S, -1, c["E"])
    allowed = (own & first[:, :, None]).any(dim=1, keepdim=True) | first[:, :, None]
    z, idx = logits.masked_fill(~allowed.expand_as(own).reshape(T, -1), -float("inf")).topk(c["k"], dim=1)
    w = torch.softmax(z, dim=1)          # the softmax over all experts, renormalised over the chosen ones
    rows = computed.reshape(-1)
    y[rows] = 0
    for e in range(c["E"] + c["ns"]):
        if e < c["E"]:
            t, j = torch.nonzero((idx == e) & rows[:, None], as_tuple=True)
            share = w[t, j]
        else:
            t = torch.nonzero(rows)[:, 0]
            share = torch.ones(t.numel(), dtype=torch.float64, device="cuda")
        if t.numel():
            a = torch.nn.functional.silu(x64[t] @ wg[e].double().T) * (x64[t] @ wu[e].double().T)
            y.index_add_(0, t, share[:, None] * (a @ wd[e].double().T))
    return y


def _accept(c, seq, pred, conf):
    """One acceptance step of a sequence (threshold 0.95): seq holds token, state and the speculated (position, token)
    pairs; pred and conf are [branches, L].  Returns the states and the confidences of the next pass's rows."""
    token, state, spec = seq["token"], seq["state"], seq["spec"]
    carries = {0: (), 1: (0,), 2: (1,), 3: (0, 1)}

    def sure(b, i):
        return i < len(spec) and pred[b, spec[i][0]] == spec[i][1] and conf[b, spec[i][0]] > np.float32(0.95)

    chain = [0]
    if sure(0, 0):
        chain += [1, 3] if sure(1, 1) else [1]
    elif sure(0, 1):
        chain += [2, 3] if sure(2, 0) else [2]
    new = {}
    for b in chain:
        held = [spec[i][0] for i in carries[b] if i < len(spec)]
        for i in carries[b]:
            if i < len(spec):
                new.setdefault(*spec[i])
        for p in range(c["block"]):
            if state[p] == W.TOK_MASKED and p not in held and conf[b, p] > np.float32(0.95):
                new.setdefault(p, int(pred[b, p]))
    state[state == W.TOK_NEW] = W.TOK_CACHED
    for p, t in new.items():
        token[p], state[p] = t, W.TOK_NEW
    last = chain[-1]
    masked = sorted(np.flatnonzero(state == W.TOK_MASKED), key=lambda p: (-conf[last, p], p))
    seq["spec"] = [(int(p), int(pred[last, p])) for p in masked[:2]] if c["branches"] == 4 else []
    states = np.tile(state, (c["branches"], 1))
    for b in range(c["branches"]):
        for i in carries[b]:
            if i < len(seq["spec"]):
                states[b, seq["spec"][i][0]] = W.TOK_NEW
    return states, np.where(states == W.TOK_MASKED, conf[last], np.float32(1))


def _attn64(c, s):
    """Every layer of an attention state: the outputs and the in-block caches after the insertion."""
    S, L, rep, d = c["seqs"], c["block"], c["n_heads"] // c["n_kv"], c["head_dim"]
    states = s["st"]["tok_state"].view(S, -1, L)
    computed = (states != W.TOK_CACHED) | (not c["flags"] & B.TEAM_F_DCD)
    out = torch.zeros(s["out"].shape, dtype=torch.float64, device="cuda")
    caches = [s["k_block"].double(), s["v_block"].double()]
    for n in range(c["layers"]):
        fresh = [s[f][n].double().view(S, -1, L, c["n_kv"], d) for f in ("k_new", "v_new")]
        for q in range(S):
            length = int(s["prefix_len"][q])
            for b in range(states.shape[1]):
                use = computed[q, b]
                k, v = (torch.cat([s[p][n, q, :length].double(), torch.where(use[:, None, None], f[q, b], cache[n, q])])
                        for p, f, cache in zip(("k_prefix", "v_prefix"), fresh, caches))
                rows = (q * states.shape[1] + b) * L + torch.nonzero(use)[:, 0]
                query = s["q"][n][rows].double().view(-1, c["n_kv"], rep, d)
                p = torch.softmax(torch.einsum("tgrd,jgd->tgrj", query, k) / d ** 0.5, dim=-1)
                out[n, rows] = torch.einsum("tgrj,jgd->tgrd", p, v).reshape(-1, c["n_heads"], d)
        keep = (computed[:, 0] & (states[:, 0] != W.TOK_MASKED))[:, :, None, None]
        for cache, f in zip(caches, fresh):
            cache[n] = torch.where(keep, f[:, 0], cache[n])
    return out, caches[0], caches[1]


def exact(case, seed):
    c = dict(case)
    s = prepare(case, seed)
    if c["kind"] == "attn":
        return _attn64(c, s)
    weights = W.device_layer_weights(_shape(c), seed, "cuda")
    y = torch.zeros(s["y"].shape, dtype=torch.float64, device="cuda")
    if c["kind"] != "decode":
        st = _step_host(c, seed)
        return _layer64(c, weights, s["x"].cuda(), st["tok_state"], st["conf"], y)
    S, nb, L = c["seqs"], c["branches"], c["block"]
    seqs = [dict(token=np.full(L, -1, np.int32), state=np.zeros(L, np.uint8), spec=[]) for _ in range(S)]
    states, conf = np.zeros((S, nb, L), np.uint8), np.zeros((S, nb, L), np.float32)
    for p in range(c["passes"]):
        y = _layer64(c, weights, s["x"][p], states, conf, y)
        pred, seen = s["pred"][p].cpu().numpy(), s["conf"][p].cpu().numpy()
        for i, q in enumerate(seqs):
            states[i], conf[i] = _accept(c, q, pred[i], seen[i])
    return (y, np.stack([q["token"] for q in seqs]), np.stack([q["state"] for q in seqs]), states.reshape(-1), conf.reshape(-1))
