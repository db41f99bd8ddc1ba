"""fp32-FMA products and attention where their tiles and splits end: partial tiles in every direction, K shorter than
a slab, K split over the warps of a CTA and over a cluster, partial key tiles, both row counts per warp."""
import numpy as np
import pytest
import torch

from oracle import rs_oracle as orc
from test_gpu_parts import ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual"])
@pytest.mark.parametrize("M,N,K", [(1, 8, 8), (31, 40, 24), (33, 32, 40), (65, 136, 96), (394, 384, 1536), (1500, 768, 768), (3000, 1536, 64), (129, 200, 776)])
def test_linear_fp32_edges(ctx, M, N, K, epilogue):   # noqa: F811
    g = torch.Generator().manual_seed(M + N + K)
    a, w, b = torch.randn(M, K, generator=g), 0.05 * torch.randn(N, K, generator=g), 0.1 * torch.randn(N, generator=g)
    res = torch.randn(M, N, generator=g) if epilogue == "residual" else None
    got = ctx.linear_fwd(a.cuda(), w.cuda(), b.cuda(), epilogue, None if res is None else res.cuda()).cpu().double().numpy()
    rows = np.arange(M) if M <= 400 else np.r_[0:130, M - 70:M]
    want = orc.linear(a.double().numpy()[rows], w.double().numpy(), b.double().numpy())
    if epilogue == "gelu":
        want = orc.gelu(want)
    if epilogue == "residual":
        want = want + res.double().numpy()[rows]
    # K fp32 roundings of partial sums of at most sum |a w|, of random sign: sqrt(K) of them, four deviations; and the
    # epilogue's few roundings of the result
    size = np.abs(a.double().numpy()[rows]) @ np.abs(w.double().numpy()).T
    bound = 2.0 ** -23 + 4 * np.sqrt(K) * 2.0 ** -24 * size + 2.0 ** -22 * np.abs(want)
    assert (np.abs(got[rows] - want) <= bound).all()
    # the bound tells fp32 products from TF32 ones (operands of 11 bits)
    if epilogue == "bias":
        tf32 = lambda t: ((t.numpy().view(np.int32) + 0x1000) & ~0x1fff).view(np.float32).astype(np.float64)   # noqa: E731
        rough = orc.linear(tf32(a)[rows], tf32(w), b.double().numpy())
        assert not (np.abs(rough - want) <= bound).all()


def test_linear_fp32_of_many_columns(ctx):   # noqa: F811
    """More than 65535 tiles of 32 columns."""
    M, N, K = 3, 2_200_008, 40
    g = torch.Generator(device="cuda").manual_seed(3)
    a, w = torch.randn(M, K, generator=g, device="cuda"), torch.randn(N, K, generator=g, device="cuda")
    got, want = ctx.linear_fwd(a, w), a.double() @ w.double().T
    assert ((got.double() - want).norm() / want.norm()).item() < 1e-6      # fp32 sums of 40 products


@pytest.mark.parametrize("M,N,K", [(1, 72, 72), (70, 200, 328), (400, 1000, 64)])       # widths the tensor cores do not take
def test_linear_bf16_on_fma_kernels(ctx, M, N, K):   # noqa: F811
    g = torch.Generator().manual_seed(M + N + K)
    a, w = torch.randn(M, K, generator=g).bfloat16(), (0.05 * torch.randn(N, K, generator=g)).bfloat16()
    assert not ctx.linear_uses_tensor_cores(torch.bfloat16, M, N, K)
    got = ctx.linear_fwd(a.cuda(), w.cuda(), None, "bias").cpu().double().numpy()
    want = orc.linear(a.double().numpy(), w.double().numpy(), np.zeros(N))
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + K * 2.0 ** -22).all()        # one bf16 rounding of the output


@pytest.mark.parametrize("B,N,H", [(1, 1, 1), (1, 15, 2), (1, 16, 1), (1, 17, 1), (2, 33, 3), (1, 63, 1), (1, 64, 2), (1, 65, 1), (2, 129, 2), (12, 97, 10), (3, 200, 40)])
def test_attention_fp32_edges(ctx, B, N, H):   # noqa: F811
    g = torch.Generator().manual_seed(N)
    qkv = torch.randn(B, N, 3, H, 64, generator=g)
    got = ctx.attn_fwd(qkv[:, :, 0].cuda(), qkv[:, :, 1].cuda(), qkv[:, :, 2].cuda()).cpu().double().numpy()
    f = qkv.double().numpy()
    want = orc.attn(f[:, :, 0], f[:, :, 1], f[:, :, 2]).reshape(B, N, H * 64)
    assert np.abs(got - want).max() < 2e-6 * np.abs(f).max()       # weights sum to one: errors of exp and of the sums, a few 2^-23 of |v|
