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


# Each weight is rounded to bf16 once and so is the output, relative errors of up to 2^-8: a sum of weights times values of independent
# signs errs by 2^-8 of their root sum of squares, which the largest errors of many outputs come near, and of any signs by 2^-8 of the sum
# of |p v|, at most |v|max.  On the average of the mantissas' squares 1 / m^2 (0.375 / ln 2, m in [1, 2) by its logarithm) an error's rms is
# 2^-8 sqrt(0.541 / 3) = 2^-8 0.425; two of them make 2.35e-3 of the outputs' rms, and 5 % more is for the samples' sake.
def _close(got, want, qkv):
    err = got.double() - want
    return err.abs().max() < 2.0 ** -8 * qkv[:, :, 2].double().abs().max() and err.norm() < 2.0 ** -8 * 0.425 * 2 ** 0.5 * 1.05 * want.norm()


# query tiles of every head with their keys cut in three, on 148 SMs: all, some and none of them
@pytest.mark.parametrize("B,H,N,cut", [(1, 1, 129, 2), (1, 2, 191, 2), (1, 12, 192, 2), (1, 12, 197, 2), (1, 3, 257, 3), (1, 5, 300, 3), (1, 4, 449, 4), (1, 4, 1000, 8),
                                       (2, 7, 1409, 0), (7, 8, 961, 1), (8, 7, 1025, 2)])
def test_keys_in_thirds(ctx, B, H, N, cut):   # noqa: F811
    import paper_2508_00367_b200 as rs
    assert rs.attn_key_cut(148, B, H, N) == cut
    assert torch.cuda.get_device_properties(0).multi_processor_count == 148
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


@pytest.mark.parametrize("B,H,N,cut", [(4, 16, 1729, 1), (2, 12, 2353, 1), (5, 3, 197, 2)])
def test_a_sample_does_not_depend_on_its_place(ctx, B, H, N, cut):   # noqa: F811
    import paper_2508_00367_b200 as rs
    assert rs.attn_key_cut(148, B, H, N) == cut
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


@pytest.mark.parametrize("B,H,N,longest,per", [(40, 2, 600, 100, 1), (60, 2, 600, 256, 2), (40, 12, 333, 333, 3), (12, 6, 1100, 1100, 3)])
@pytest.mark.parametrize("gain", [1.0, 8.0])
def test_counts_per_sample_sorted(ctx, B, H, N, longest, per, gain):   # noqa: F811
    """The kernel that sorts the samples, one, two and three query tiles to an item (by the tiles that the counts leave), with scores that
    raise the running maximum in many key tiles and scores that do not."""
    import paper_2508_00367_b200 as rs
    assert rs.attn_kernel_choice(148, B, H, N, counts=True) == 3
    g = torch.Generator(device="cuda").manual_seed(longest)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda")
    qkv[:, :, 0] *= gain
    qkv[:, :, 1] *= torch.linspace(0.3, 1.7, N, device="cuda")[None, :, None, None]     # later keys reach higher
    qkv = qkv.bfloat16()
    lens = torch.randint(1, longest + 1, (B,), generator=g, device="cuda").to(torch.int32)
    lens[1] = longest
    assert min(-(-int(((lens + 127) // 128).sum()) * H // 148), 3) == per
    got = ctx.attn_fwd_ragged(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], lens)
    ctx.async_status()
    for b in range(0, B, 1 if B < 20 else 3):
        n = int(lens[b])
        err = got[b:b + 1, :n].double() - _reference(qkv[b:b + 1, :n])
        assert err.abs().max() < 2.0 ** -8 * qkv[b, :n, 2].double().abs().max(), (b, n)


@pytest.mark.parametrize("counts", ["equal", "one key tile apart", "one long"])
def test_every_sample_of_a_sorted_batch(ctx, counts):   # noqa: F811
    """256 samples, the most that are sorted, and ties in their order: every row of every sample is written, once, with its own sample's result."""
    B, H, N = 256, 3, 197
    g = torch.Generator(device="cuda").manual_seed(B)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    lens = {"equal": torch.full((B,), 150), "one key tile apart": torch.arange(B) % 4 * 64 + 1, "one long": torch.tensor([1] * (B - 1) + [N])}[counts].to(torch.int32).cuda()
    got = ctx.attn_fwd_ragged(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], lens, out=torch.full((B, N, H * 64), float("nan"), dtype=torch.bfloat16, device="cuda"))
    ctx.async_status()
    q, k, v = (qkv[:, :, i].transpose(1, 2).double() for i in range(3))
    past = torch.arange(N, device="cuda")[None] >= lens[:, None]
    s = (q @ k.transpose(2, 3) / 8.0).masked_fill(past[:, None, None], float("-inf"))
    want = (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(B, N, -1).masked_fill(past[..., None], 0.0)
    assert _close(got, want, qkv)


@pytest.mark.parametrize("B", [74, 75])
@pytest.mark.parametrize("H", [1, 2, 3, 4])
def test_tiles_to_an_item_of_a_sorted_batch(ctx, B, H):   # noqa: F811
    """Two query tiles per head: as many as fill one, two, three and four rounds of 148, and a sample more, on both sides of where one, two or
    three go to an item."""
    import paper_2508_00367_b200 as rs
    N = 600
    assert rs.attn_kernel_choice(148, B, H, N, counts=True) == 3
    g = torch.Generator(device="cuda").manual_seed(B + H)
    qkv = torch.randn(B, N, 3, H, 64, generator=g, device="cuda").bfloat16()
    lens = (129 + torch.arange(B) * 50 % 128).to(torch.int32).cuda()
    got = ctx.attn_fwd_ragged(qkv[:, :, 0], qkv[:, :, 1], qkv[:, :, 2], lens)
    ctx.async_status()
    for b in range(0, B, 3):
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
