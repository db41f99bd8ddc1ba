"""Selection and row gather at the edges of their launch rules: keys per thread change after 1024, 2048, 5120 and
16384 tokens; rows of up to 32 and 64 sixteen-byte pieces are moved several to a warp."""
import numpy as np
import pytest
import torch

from oracle import rs_oracle as orc
from test_gpu_parts import _scores, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["normal", "ties", "special", "equal"])
@pytest.mark.parametrize("N", [2048, 2049, 5120, 5121, 16384, 16385])
def test_selection_at_the_keys_per_thread_edges(ctx, kind, N):   # noqa: F811
    s = _scores(2, N, kind, N)
    for has_cls in (True, False):
        for r in (1, N // 3, N - 2, N - 1):
            _, keep = ctx.topk_compact(torch.from_numpy(s).cuda(), None, r, has_cls)
            np.testing.assert_array_equal(keep.cpu().numpy(), orc.topk(s.astype(np.float64), r, has_cls), err_msg=f"r={r} cls={has_cls}")


@pytest.mark.parametrize("kind", ["normal", "ties"])
@pytest.mark.parametrize("N", [2560, 2561, 5120])
def test_selection_of_many_samples(ctx, kind, N):   # noqa: F811
    """Two samples to an SM and more: sixteen keys per thread from 2561 tokens on."""
    B = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    s = _scores(B, N, kind, N)
    _, keep = ctx.topk_compact(torch.from_numpy(s).cuda(), None, N // 3, True)
    np.testing.assert_array_equal(keep.cpu().numpy(), orc.topk(s.astype(np.float64), N // 3, True))


@pytest.mark.parametrize("pieces", [1, 31, 32, 33, 63, 64, 65, 300])
@pytest.mark.parametrize("B,N,r", [(1, 3, 1), (3, 50, 7), (62, 130, 7)])       # row counts that leave a warp partly filled; the last: several to a warp
def test_rows_of_every_width_class(ctx, pieces, B, N, r):   # noqa: F811
    D = 8 * pieces
    s = _scores(B, N, "normal", pieces)
    x = torch.randn(B, N, D, generator=torch.Generator().manual_seed(pieces)).bfloat16()
    buf = torch.full((B * (N - r) * D + 128,), -7.0, dtype=torch.bfloat16, device="cuda")      # canaries around the rows
    xo = buf[64:-64].view(B, N - r, D)
    _, keep = ctx.topk_compact(torch.from_numpy(s).cuda(), x.cuda(), r, True, x_out=xo)
    want = orc.topk(s.astype(np.float64), r, True)
    np.testing.assert_array_equal(keep.cpu().numpy(), want)
    assert torch.equal(xo.cpu(), torch.stack([x[b][torch.from_numpy(want[b]).long()] for b in range(B)]))
    assert (buf[:64] == -7).all() and (buf[-64:] == -7).all()


@pytest.mark.parametrize("dist", ["l2", "l1", "cos"])
@pytest.mark.parametrize("pieces", [1, 2, 3, 16, 17, 32, 33, 64, 65])
def test_score_of_every_width_class(ctx, pieces, dist):   # noqa: F811
    D, rows = 8 * pieces, 131                                   # a row count that leaves a warp partly filled
    g = torch.Generator().manual_seed(pieces)
    a, b = torch.randn(1, rows, D, generator=g).bfloat16(), torch.randn(1, rows, D, generator=g).bfloat16()
    buf = torch.full((rows + 2,), -7.0, device="cuda")
    got = ctx.shift_score(a.cuda(), b.cuda(), dist, out=buf[1:-1].view(1, rows))
    want = orc.shift_score(a.double().numpy(), b.double().numpy(), dist)
    if dist == "cos":
        np.testing.assert_allclose(got.cpu().double().numpy(), want, rtol=0, atol=2e-6)    # 1 - cos cancels: an absolute bound
    else:
        np.testing.assert_allclose(got.cpu().double().numpy(), want, rtol=2e-6, atol=0)    # fp32 sum of D <= 520 terms
    assert buf[0] == -7 and buf[-1] == -7


@pytest.mark.parametrize("pieces", [2, 3, 32, 33, 64, 65])
@pytest.mark.parametrize("H,W,dr,dc", [(7, 5, 2, 1), (90, 91, 30, 40), (91, 91, 1, 90), (91, 90, 1, 3)])   # staged scores up to 8192; the last: several to a warp
def test_grid_rows_of_every_width_class(ctx, pieces, H, W, dr, dc):   # noqa: F811
    D = 8 * pieces
    s = _scores(2, H * W, "normal", pieces).reshape(2, H, W)
    x = torch.randn(2, H, W, D, generator=torch.Generator().manual_seed(pieces)).bfloat16()
    xo, kr, kc = ctx.linewise_compact(torch.from_numpy(s).cuda(), x.cuda(), dr, dc)
    want_r, want_c = orc.linewise(s.astype(np.float64), dr, dc)
    np.testing.assert_array_equal(kr.cpu().numpy(), want_r)
    np.testing.assert_array_equal(kc.cpu().numpy(), want_c)
    for b in range(2):
        assert torch.equal(xo[b].cpu(), x[b][torch.from_numpy(want_r[b]).long()][:, torch.from_numpy(want_c[b]).long()])


@pytest.mark.parametrize("dist", ["l2", "l1", "cos"])
@pytest.mark.parametrize("D,edge", [(8, 2960), (24, 5920), (128, 5920), (136, 14800), (256, 14800), (264, 1480), (512, 1480)])
def test_scores_where_several_tokens_share_a_warp(ctx, D, edge, dist):   # noqa: F811
    """The token counts (on 148 SMs) from which tokens of up to 64 pieces go several to a warp, one and a warp's worth more."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for T in (edge * sms // 148, edge * sms // 148 + 1, edge * sms // 148 + 129):
        g = torch.Generator(device="cuda").manual_seed(T)
        a, b = (torch.randn(1, T, D, generator=g, device="cuda").bfloat16() for _ in range(2))
        got, u, v = ctx.shift_score(a, b, dist=dist).double(), a.double(), b.double()
        want = (u - v).norm(dim=-1) if dist == "l2" else (u - v).abs().sum(-1) if dist == "l1" else 1 - (u * v).sum(-1) / (u.norm(dim=-1) * v.norm(dim=-1))
        # sums of at most 512 terms in fp32; the cosine is a difference of numbers near one
        assert (got - want).abs().max() <= (2e-6 if dist == "cos" else 2e-6 * want.max())


def _needs_memory(nbytes):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < nbytes:
        pytest.skip("not enough free device memory")


def test_more_kept_rows_than_a_launch_counts(ctx):   # noqa: F811
    """2^31 kept rows and more: the samples around the place where the second launch begins, the first and the last."""
    N, r, D = 32768, 1, 8
    K = N - r
    cut = (2 ** 31 - 1) // K                                         # samples of the first launch
    B = cut + 3
    _needs_memory(100 << 30)
    x, s = torch.empty(B, N, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(B, N, device="cuda")
    look = [0, 1, cut - 1, cut, cut + 1, B - 1]
    x[look] = torch.randn(len(look), N, D, device="cuda").bfloat16()
    for i, b in enumerate(look):
        s[b, 5 + i] = -1.0                                           # the token that goes
    x_out, keep = ctx.topk_compact(s, x, r)
    for i, b in enumerate(look):
        want = [t for t in range(N) if t != 5 + i]
        assert keep[b].tolist() == want and torch.equal(x_out[b], x[b, want])
    del x, s, x_out, keep
    torch.cuda.empty_cache()


def test_more_kept_positions_than_a_launch_counts(ctx):   # noqa: F811
    H = W = 256
    D, dr, dc = 8, 1, 0
    cut = (2 ** 31 - 1) // ((H - dr) * (W - dc))
    B = cut + 2
    _needs_memory(100 << 30)
    x, s = torch.empty(B, H, W, D, dtype=torch.bfloat16, device="cuda"), torch.ones(B, H, W, device="cuda")
    look = [0, cut - 1, cut, B - 1]
    x[look] = torch.randn(len(look), H, W, D, device="cuda").bfloat16()
    for i, b in enumerate(look):
        s[b, 7 + i] = 0.0                                            # the line that goes
    x_out, rows, cols = ctx.linewise_compact(s, x, dr, dc)
    for i, b in enumerate(look):
        want = [t for t in range(H) if t != 7 + i]
        assert rows[b].tolist() == want and cols[b].tolist() == list(range(W)) and torch.equal(x_out[b], x[b, want])
    del x, s, x_out, rows, cols
    torch.cuda.empty_cache()
