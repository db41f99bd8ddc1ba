"""Attention weights over the whole range of the exponential: rows whose scores lie up to hundreds of octaves below
their maximum, maxima that rise from key tile to key tile, and sums of very many small weights."""
import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from test_gpu_parts import ctx, pinned   # noqa: F401  (the module's context fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("gain", [0.02, 1.0, 8.0, 30.0])
def test_weights_over_the_range_of_exp2(pinned, kernel, gain):   # noqa: F811
    B, N, H = 1, 450, 2
    g = torch.Generator().manual_seed(int(gain * 100))
    qkv = torch.randn(B, N, 3, H, 64, generator=g)
    qkv[:, :, 0] *= gain                                         # scores with a standard deviation of `gain` nats
    qkv[:, :, 1] *= torch.linspace(0.3, 1.7, N)[None, :, None, None]     # later keys reach higher
    qkv = qkv.to(torch.bfloat16)
    dq = qkv.cuda()
    got = pinned[kernel].attn_fwd(dq[:, :, 0], dq[:, :, 1], dq[:, :, 2]).cpu().double().numpy()
    f = qkv.double().numpy()
    want = orc.attn(f[:, :, 0], f[:, :, 1], f[:, :, 2]).reshape(B, N, H * 64)
    # weights rounded to bf16 (2^-9 each, they sum to one), values up to |v|max; one rounding of the output
    assert np.abs(got - want).max() < (2.0 ** -8) * np.abs(f[:, :, 2]).max()


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
def test_scores_that_are_not_finite(pinned, kernel, value):   # noqa: F811
    """A key whose score is NaN or +inf makes the rows NaN at whatever column of a key tile it stands, whole tile or
    partial; one at -inf has weight zero.  Sample b has that key at position where[b]."""
    N, H = 400, 1
    where = torch.cat([torch.arange(0, 192), torch.arange(384, 400)])
    B = len(where)
    g = torch.Generator(device="cuda").manual_seed(7)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    qkv[:, :, 0, :, 0] = 1.0
    qkv[torch.arange(B), where, 1, :, 0] = value
    got = pinned[kernel].attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2]).double()
    if value != float("-inf"):
        assert got.isnan().all(), where[~got.isnan().flatten(1).all(1).cpu()]
        return
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    want = (torch.softmax(q @ k.transpose(2, 3) / 8.0, -1) @ v).transpose(1, 2).reshape(B, N, H * 64)
    assert (got - want).abs().max() < 2.0 ** -8 * v.abs().max()      # as below


@pytest.mark.parametrize("B,H,N", [(1, 2, 129), (3, 1, 200), (40, 20, 133), (25, 9, 256), (13, 12, 300), (30, 12, 500), (2, 3, 600), (11, 16, 577)])
def test_query_tiles_across_heads(pinned, B, H, N):   # noqa: F811
    """Three query tiles to an item, over the ends of heads and samples: two to five tiles per head, whole rounds of
    items with tiles of the last round handed out singly or in threes."""
    g = torch.Generator(device="cuda").manual_seed(N)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    got = pinned[3].attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2]).double()
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    want = torch.softmax(q @ k.transpose(2, 3) / 8.0, -1) @ v
    # weights rounded to bf16 (2^-9 each, they sum to one), values up to |v|max; one rounding of the output
    assert (got - want.transpose(1, 2).reshape(B, N, H * 64)).abs().max() < 2.0 ** -8 * v.abs().max()


@pytest.mark.parametrize("B,H,N,counts", [(8, 12, 129, False), (8, 12, 197, False), (4, 16, 300, False), (2, 12, 2353, False),
                                          (64, 3, 101, False), (30, 12, 300, True), (3, 3, 200, True)])
@pytest.mark.parametrize("where", [70, 100, 127, 128])
def test_the_largest_weight_is_not_rounded(ctx, B, H, N, counts, where):   # noqa: F811
    """One key outweighs the rest by 3 to 5 nats (less than what raises the running maximum) and is the only one with values, so the
    output is its share p of the weights times its value.  Its weight is exact, or rounded the same above and below the line: an
    error e of it leaves e (1 - p), 1 - p <= 0.05, which changes the bf16 of at most 5 % of the outputs (all of e would: half)."""
    if where >= N:
        return
    g = torch.Generator(device="cuda").manual_seed(where + N)
    q, k, v = (torch.zeros(B, N, H, 64, device="cuda") for _ in range(3))
    a = torch.rand(B, N, H, generator=g, device="cuda").mul_(2).add_(3).bfloat16()
    q[..., 0], q[..., 1] = a.float(), 8.0
    k[..., 1] = -12.0                                            # scores of -12 nats,
    k[:, 3, :, 1] = 0.0                                          # one of 0
    k[:, where, :, 0], k[:, where, :, 1] = 8.0, 0.0              # and one of a
    v[:, where] = torch.rand(B, H, 64, generator=g, device="cuda").add_(1).bfloat16().float()
    q, k, v = q.bfloat16(), k.bfloat16(), v.bfloat16()
    lens = torch.randint(max(130, where + 1), N + 1, (B,), generator=g, device="cuda").to(torch.int32) if counts else torch.full((B,), N, device="cuda")
    got = (ctx.attn_fwd_ragged(q, k, v, lens) if counts else ctx.attn_fwd(q, k, v)).view(B, N, H, 64)
    w = a.double().exp()
    p = w / (w + 1 + (lens.view(B, 1, 1) - 2) * np.exp(-12.0))
    want = (p[..., None] * v[:, where].double()[:, None]).bfloat16()
    # (2353: without the query tiles at the end that are cut by keys, which have a running maximum per part instead)
    used = (torch.arange(N, device="cuda")[None] < lens.clamp(max=2048)[:, None])[:, :, None, None].expand_as(got)
    if where < 128 or not counts or B > 3:                       # (small batches with counts: the kernel that knows no true maximum)
        assert (got != want)[used].double().mean() < 0.05
    assert ((got.float() - want.float()).abs() <= want.float() * 2.0 ** -7)[used].all()


@pytest.mark.parametrize("B,H,N", [(1, 2, 197), (4, 6, 197), (1, 12, 577), (30, 12, 300)])
@pytest.mark.parametrize("last", [64, 128, 150])
def test_first_keys_without_weight(ctx, pinned, B, H, N, last):   # noqa: F811
    """Keys at -infinity that fill the first key tile (or tiles) are weights of zero in every kernel: both on the tensor cores, with and
    without counts, and the fp32 one with one group of warps and with four."""
    g = torch.Generator(device="cuda").manual_seed(last + N)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    qkv[:, :, 0, :, 0] = 1.0
    qkv[:, :last, 1, :, 0] = float("-inf")
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    want = (torch.softmax(q @ k.transpose(2, 3) / 8.0, -1) @ v).transpose(1, 2).reshape(B, N, H * 64)
    bound = 2.0 ** -8 * v.abs().max()                                # as above
    a = [qkv[:, :, i] for i in range(3)]
    lens = torch.full((B,), N, dtype=torch.int32, device="cuda")
    for c in (ctx, pinned[2], pinned[3]):
        assert (c.attn_fwd(*a).double() - want).abs().max() < bound
        assert (c.attn_fwd_ragged(*a, lens).double() - want).abs().max() < bound
    assert (ctx.attn_fwd(*(t.float() for t in a)).double() - want).abs().max() < 2e-6 * v.abs().max()     # (errors of exp and of the sums)
