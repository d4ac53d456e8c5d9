"""The tensor-core router (bf16 activations, more than 8 rows) against the oracle's fp64 dot products, at the edges of its
tiles: ragged rows and experts, hidden sizes that leave warps without a block, every tile size of its dispatch."""
import numpy as np
import pytest
import torch

from oracle import team_oracle as O
from paper_2602_08404_b200 import binding as B
from tests import _parity as P

pytestmark = pytest.mark.gpu


def _route(x, w_router, k):
    T, H = x.shape
    E = w_router.shape[0]
    cfg = B.make_config(H, E, k, 64, max_rows=T, max_groups=1, dtype=B.TEAM_DTYPE_BF16)
    ctx = B.team_create(cfg)
    gu, dn = (torch.zeros(m * E * 64 * H, dtype=torch.bfloat16, device="cuda") for m in (2, 1))
    B.team_set_weights(ctx, w_router, w_gu_tiles=gu, w_down_tiles=dn)
    st = dict(tok_state=torch.zeros(T, dtype=torch.uint8, device="cuda"), conf=torch.zeros(T, device="cuda"),
              **{n: torch.zeros(T, dtype=torch.int32, device="cuda") for n in ("pos", "group", "branch")})
    out = {n: v for n, v in B.alloc_routing(cfg, T).items() if n in ("probs", "topk_idx", "topk_w", "margin")}
    B.team_route(ctx, x, st, out)
    got = B.routing_to_host(out)
    B.team_destroy(ctx)
    return got


@pytest.mark.parametrize("T,H,E", [(9, 128, 9), (16, 2048, 128), (17, 1536, 97), (65, 1024, 33), (185, 1536, 96), (256, 2176, 129),
                                   (300, 640, 250), (1000, 384, 100), (2048, 256, 128), (2047, 128, 256)])
def test_logits_of_every_tile_size(T, H, E):
    g = torch.Generator().manual_seed(T + H)
    x = torch.randn((T, H), generator=g).to(torch.bfloat16)
    w = torch.randn((E, H), generator=g) / H ** 0.5
    k = min(8, E - 1)
    got = _route(x.cuda(), w.cuda(), k)
    logits, probs = O.router(x.float().numpy(), w.numpy())
    # a logit is off by at most a few roundings of its partial sums (2^-24 each): PROBS_ATOL holds with room to spare
    np.testing.assert_allclose(got["probs"], probs, rtol=0, atol=P.PROBS_ATOL)
    clear = 0
    for t in range(T):
        take, _ = O.topk_row(logits[t], k)
        if P.ordering_margin(logits[t], take, range(E)) > P.MARGIN:
            assert got["topk_idx"][t].tolist() == list(take), t
            clear += 1
    assert clear > 0.9 * T


def test_infinite_and_large_weights_keep_their_sums():
    """The remainder of an infinity is not a number: such logits are formed without splitting, as plain fp32 sums."""
    T, H, E = 20, 256, 24
    g = torch.Generator().manual_seed(3)
    x = torch.randn((T, H), generator=g).to(torch.bfloat16)
    x[:, 5] = x[:, 5].abs() + 0.5
    w = torch.randn((E, H), generator=g) / H ** 0.5
    w[11, 5] = float("inf")
    w[12, 5] = -float("inf")
    w[13, 5] = 3.4e38                     # rounds up to infinity in bf16, is cut to a finite number in two parts
    x[0, 5] = 0.5
    got = _route(x.cuda(), w.cuda(), 2)
    assert (got["topk_idx"][:, 0] == 11).all()
    assert not (got["topk_idx"] == 12).any()
    assert (got["topk_idx"][:, 1] == 13).all()
    assert got["margin"][0] > 1e37        # row 0: 0.5 * 3.4e38 is finite and above the third choice by that much


def test_rows_that_are_only_8_byte_aligned():
    """team_route takes bf16 rows at 8-byte alignment, with every tile size of its dispatch: the same sums as for aligned
    rows.  What no load width fits is an argument error."""
    for T, H, E in [(4, 256, 16), (9, 2048, 24), (65, 384, 33), (300, 640, 100), (1000, 256, 128), (2048, 128, 256)]:
        g = torch.Generator().manual_seed(T)
        x = torch.randn((T, H), generator=g).to(torch.bfloat16).cuda()
        w = (torch.randn((E, H), generator=g) / H ** 0.5).cuda()
        shifted = torch.zeros(T * H + 4, dtype=torch.bfloat16, device="cuda")[4:].view(T, H)
        shifted.copy_(x)
        assert x.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 == 8
        a, b = _route(x, w, 4), _route(shifted, w, 4)
        if T > 8:
            for n in a:
                np.testing.assert_array_equal(a[n], b[n], err_msg=f"{n} {T}")
        else:                             # aligned rows run the FMA kernel
            np.testing.assert_allclose(a["probs"], b["probs"], rtol=0, atol=P.PROBS_ATOL)
        odd = torch.zeros(T * H + 2, dtype=torch.bfloat16, device="cuda")[2:].view(T, H)
        with pytest.raises(B.TeamError):
            _route(odd, w, 4)


def test_fp32_rows_need_16_bytes():
    cfg = B.make_config(64, 8, 2, 16, max_rows=4, dtype=B.TEAM_DTYPE_F32)
    ctx = B.team_create(cfg)
    w = [torch.zeros(s, device="cuda") for s in ((8, 64), (8, 16, 64), (8, 16, 64), (8, 64, 16))]
    B.team_set_weights(ctx, *w)
    st = dict(tok_state=torch.zeros(4, dtype=torch.uint8, device="cuda"), conf=torch.zeros(4, device="cuda"),
              **{n: torch.zeros(4, dtype=torch.int32, device="cuda") for n in ("pos", "group", "branch")})
    with pytest.raises(B.TeamError):
        B.team_route(ctx, torch.zeros(4 * 64 + 2, device="cuda")[2:].view(4, 64), st, dict(topk_idx=torch.zeros((4, 2), dtype=torch.int32, device="cuda")))
    B.team_destroy(ctx)


def _time_route(ctx, x, st, out):
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    best = float("inf")
    for _ in range(20):
        ev[0].record()
        for _ in range(10):
            B.team_route(ctx, x, st, out)
        ev[1].record()
        ev[1].synchronize()
        best = min(best, ev[0].elapsed_time(ev[1]) * 100)
    return best


def test_activations_that_are_not_finite_stay_in_their_rows():
    """Rows of NaN and infinities: the other rows' results do not change by a bit; the x of cached rows is not used under
    delayed caching, so whatever it holds costs nothing either."""
    T, H, E, k = 300, 4096, 128, 4
    g = torch.Generator().manual_seed(8)
    x = torch.randn((T, H), generator=g).to(torch.bfloat16).cuda()
    w = (torch.randn((E, H), generator=g) / H ** 0.5).cuda()
    cfg = B.make_config(H, E, k, 64, max_rows=T, dtype=B.TEAM_DTYPE_BF16, flags=B.TEAM_F_DCD)
    ctx = B.team_create(cfg)
    gu, dn = (torch.zeros(m * E * 64 * H, dtype=torch.bfloat16, device="cuda") for m in (2, 1))
    B.team_set_weights(ctx, w, w_gu_tiles=gu, w_down_tiles=dn)
    state = torch.zeros(T, dtype=torch.uint8)
    state[50:250] = B.TEAM_TOK_CACHED
    st = dict(tok_state=state.cuda(), conf=torch.zeros(T, device="cuda"),
              **{n: torch.zeros(T, dtype=torch.int32, device="cuda") for n in ("pos", "group", "branch")})
    out = {n: v for n, v in B.alloc_routing(cfg, T).items() if n in ("probs", "topk_idx", "topk_w", "margin")}
    B.team_route(ctx, x, st, out)
    want = B.routing_to_host(out)
    finite_us = _time_route(ctx, x, st, out)
    bad = x.clone()
    bad[50:150] = float("nan")
    bad[150:250, 7] = float("inf")
    B.team_route(ctx, bad, st, out)
    got = B.routing_to_host(out)
    for n in want:
        np.testing.assert_array_equal(got[n], want[n], err_msg=n)
    # a logit formed again is a chain of 4096 dependent steps, twice the rest of the call
    assert _time_route(ctx, bad, st, out) < 1.25 * finite_us
    bad[0], bad[17, 5], bad[299, 4000] = float("nan"), float("inf"), -float("inf")
    B.team_route(ctx, bad, st, out)
    got = B.routing_to_host(out)
    rest = np.setdiff1d(np.arange(T), [0, 17, 299])
    for n in want:
        np.testing.assert_array_equal(got[n][rest], want[n][rest], err_msg=n)
    assert np.isnan(got["probs"][[0, 17, 299]]).all()
    # an infinite activation makes a logit infinite with the sign of its weight, as a plain fp32 sum does
    assert set(got["topk_idx"][17].tolist()) <= set(torch.nonzero(w[:, 5].cpu() > 0)[:, 0].tolist())
    B.team_destroy(ctx)
