"""team_moe_forward_host with blocks on either side of what it copies by kernel: both directions by kernel, x by kernel and y by
the copy engine, both by the copy engine; fewer rows than the context holds, and another row count on every call (the recorded
step is recorded anew)."""
import pytest
import torch

from paper_2602_08404_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [True, False], ids=["own_stream", "default_stream"])
@pytest.mark.parametrize("dtype", [B.TEAM_DTYPE_BF16, B.TEAM_DTYPE_F32], ids=["bf16", "f32"])
def test_copies_of_every_size(dtype, own_stream):
    H, E, k, I, most = (2048, 12, 3, 64, 600) if dtype == B.TEAM_DTYPE_BF16 else (1024, 12, 3, 32, 600)
    g = torch.Generator().manual_seed(5)
    f = torch.bfloat16 if dtype == B.TEAM_DTYPE_BF16 else torch.float32
    wr = (torch.randn((E, H), generator=g) / H ** 0.5).cuda()
    wg, wu, wd = ((0.02 * torch.randn(s, generator=g)).to(f).cuda() for s in ((E, I, H), (E, I, H), (E, H, I)))
    cfg = B.make_config(H, E, k, I, max_rows=most, max_groups=1, dtype=dtype, flags=B.TEAM_F_DCD | B.TEAM_F_LAC)
    ctxs = [B.team_create(cfg) for _ in range(2)]
    weights = dict(zip(("w_gu_tiles", "w_down_tiles"), B.team_pack_w_tiles(wg, wu, wd))) if dtype == B.TEAM_DTYPE_BF16 else \
        dict(w_gate=wg, w_up=wu, w_down=B.team_pack_w_down(wd))
    for ctx in ctxs:
        B.team_set_weights(ctx, wr, **weights)
    y_dev = torch.zeros((most, H), device="cuda")
    stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for T in (5, 5, 200, 600, 257, 200, 1, 600, 5):
            x = torch.randn((T, H), generator=g).to(f)
            at = torch.arange(T)
            st = dict(tok_state=torch.randint(0, 3, (T,), generator=g, dtype=torch.uint8), conf=torch.rand(T, generator=g),
                      pos=(at % 8).to(torch.int32), group=torch.zeros(T, dtype=torch.int32), branch=(at // 8).to(torch.int32))
            y_host = torch.full((T, H), 7.0)
            B.team_moe_forward(ctxs[0], x.cuda(), {n: v.cuda() for n, v in st.items()}, None, y_dev[:T])
            B.team_moe_forward_host(ctxs[1], x, st, None, y_host)
            ref = y_dev[:T].cpu()
            # the fp32 reductions of the experts arrive in another order: equal to rounding of the sums
            assert torch.allclose(y_host, ref, rtol=0, atol=1e-5 * float(ref.abs().max())), T
            for ctx in ctxs:
                assert B.team_read_status(ctx)[0] == B.TEAM_OK
    for ctx in ctxs:
        B.team_destroy(ctx)
