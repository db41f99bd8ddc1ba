"""Attention with the keys of a query tile cut in three (few query tiles, or some of every head's), whole and partial key
tiles, thirds of unequal length and empty ones, and batches with a count per sample on either side of the kernel's limit."""
import pytest
import torch

from test_gpu_parts import ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


def _reference(qkv):
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    s = (q @ k.transpose(2, 3) / 8.0)
    return (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(qkv.shape[0], qkv.shape[1], -1)


# weights rounded to bf16 (2^-9 each, they sum to one), values up to |v|max; one rounding of the output
def _close(got, want, qkv):
    return (got.double() - want).abs().max() < 2.0 ** -8 * qkv[:, :, 2].double().abs().max()


@pytest.mark.parametrize("B,H,N", [(1, 1, 129), (1, 2, 191), (1, 12, 192), (1, 12, 197), (1, 3, 257), (1, 5, 300), (1, 4, 449), (1, 4, 1000), (2, 7, 1409)])
def test_keys_in_thirds(ctx, B, H, N):   # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(N)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    got = ctx.attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2])
    ctx.async_status()
    assert _close(got, _reference(qkv), qkv)


@pytest.mark.parametrize("N", [197, 449])
@pytest.mark.parametrize("first,last", [(0, 64), (0, 130), (64, 192), (128, 197)])
def test_a_third_without_weight(ctx, N, first, last):   # noqa: F811
    """Keys at -infinity that fill whole key tiles, the first of a third among them: weights of zero."""
    g = torch.Generator(device="cuda").manual_seed(first)
    qkv = torch.randn(1, N, 3, 2, 64, generator=g, device="cuda").bfloat16()
    qkv[:, :, 0, :, 0] = 1.0
    qkv[:, first:last, 1, :, 0] = float("-inf")
    got = ctx.attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2])
    assert _close(got, _reference(qkv), qkv)


@pytest.mark.parametrize("B,H,N", [(4, 16, 1729), (2, 12, 2353), (5, 3, 197)])
def test_a_sample_does_not_depend_on_its_place(ctx, B, H, N):   # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(N)
    qkv = torch.randn(1, N, 3, H, 64, generator=g, device="cuda").bfloat16().repeat(B, 1, 1, 1, 1)
    got = ctx.attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2])
    assert all(torch.equal(got[b], got[0]) for b in range(1, B))
    assert _close(got[:1, -300:], _reference(qkv[:1])[:, -300:], qkv)


@pytest.mark.parametrize("B", [1, 7, 70, 256, 257])
def test_counts_per_sample(ctx, B):   # noqa: F811
    N, H = 200, 3
    g = torch.Generator(device="cuda").manual_seed(B)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    lens = torch.randint(1, N + 1, (B,), generator=g, device="cuda").to(torch.int32)
    lens[-1] = N
    got = ctx.attn_fwd_ragged(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], lens)
    ctx.async_status()
    for b in range(0, B, 1 if B < 10 else 11):
        n = int(lens[b])
        assert _close(got[b:b + 1, :n], _reference(qkv[b:b + 1, :n]), qkv[b:b + 1, :n]), (b, n)


@pytest.mark.parametrize("B,H,N", [(1, 3, 65), (1, 1, 127), (1, 2, 200), (1, 3, 257), (1, 9, 256), (2, 6, 197), (1, 2, 600)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_fp32_key_tiles_in_groups(ctx, B, H, N, dtype):   # noqa: F811
    """The fp32-FMA kernel with its key tiles dealt out to four groups of warps (few query rows), a group without a tile among
    them; bf16 takes that kernel with strides that tensor maps cannot express only, so a context without tensor cores runs it."""
    import os
    import paper_2508_00367_b200 as rs
    c = ctx
    if dtype == torch.bfloat16:
        os.environ["RS_DISABLE_TC"] = "1"
        try:
            c = rs.Context(0)
        finally:
            del os.environ["RS_DISABLE_TC"]
    g = torch.Generator(device="cuda").manual_seed(N)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").to(dtype)
    qkv[:, :, 0, :, 0] = 1.0
    if N > 128:
        qkv[:, 64:128, 1, :, 0] = float("-inf")                  # a group's only tile without weight
    got = c.attn_fwd(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2])
    # fp32: errors of exp and of the sums, a few 2^-23 of |v| (the weights sum to one); bf16: one rounding of the output
    bound = (2e-6 if dtype == torch.float32 else 2.0 ** -8) * qkv[:, :, 2].double().abs().max()
    assert (got.double() - _reference(qkv)).abs().max() < bound
    if c is not ctx:
        c.close()
