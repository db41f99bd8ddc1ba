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
