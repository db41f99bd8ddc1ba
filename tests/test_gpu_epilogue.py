"""Epilogues of the tensor-core products: GELU over its range and at values that are not finite, and every score at row
counts that stay with the pair-tile kernel (a last row tile of nine rows, output in both types)."""
import math

import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from paper_2508_00367_b200 import synth
from test_gpu_block import _np, _run_block, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [130, 16500])
def test_gelu_range(ctx, M):   # noqa: F811
    v = torch.linspace(-9.0, 9.0, M * 128).reshape(M, 128).bfloat16()
    v[0, :8] = torch.tensor([0.0, -0.0, 30.0, -30.0, 1e4, -1e4, 3e38, -3e38]).bfloat16()
    b = torch.zeros(128)
    b[125], b[126], b[127] = math.inf, -math.inf, math.nan
    got = ctx.linear_fwd(v.cuda(), torch.eye(128).bfloat16().cuda(), b.cuda(), "gelu").cpu().double()
    want = orc.gelu(v.double().numpy())
    # half a unit in the last place of a bf16 (8 significant bits: 2^-8 of the value at most), and 1e-6 of the polynomial
    err = np.abs(got.numpy() - want)[:, :125] - 2.0 ** -8 * np.abs(want[:, :125])
    assert err.max() < 1e-6, err.max()
    assert (got[:, 125] == math.inf).all() and (got[:, 126] == 0).all() and got[:, 127].isnan().all()


@pytest.mark.parametrize("out", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("mode,dist", [("mlp", "l2"), ("mlp", "cos"), ("mlp_delta", "l1"), ("attn", "l1"), ("attn", "cos"), ("block", "l2")])
def test_block_pair_tiles_every_score(ctx, mode, dist, out):   # noqa: F811
    B, N, D, H, r = 9, 257, 384, 6, 40
    x, w = synth.make_tokens(B, N, D, "bf16", seed=11), synth.make_block_weights(D, 4 * D, "bf16", seed=12)
    ref = orc.block_fwd(x.double().numpy(), _np(w), H, r, score_mode=mode, dist=dist)
    res = _run_block(ctx, x, w, H, r, "bf16", out, score_mode=mode, dist=dist)
    rounded = out == torch.bfloat16
    parity.check_float(res["x_full"].double().numpy(), orc.round_to(ref["x_hat"], "bf16") if rounded else ref["x_hat"], "bf16", rounded)
    # 5e-4 where the exact x' dominates the distance, else sums of bf16-operand products alone; |m| is a tenth of |x'|
    tol = 5e-4 if (mode, dist) == ("mlp", "l2") else 3e-3 if mode == "mlp_delta" else 2e-3
    rel = np.abs(res["scores"].double().numpy() - ref["scores"]) / np.abs(ref["scores"])
    assert rel.max() < tol, rel.max()


@pytest.mark.parametrize("D", [128, 192, 256, 384])
@pytest.mark.parametrize("B,N", [(1, 1), (1, 31), (3, 33), (5, 130)])
def test_block_narrow_layernorm_rows(ctx, B, N, D):   # noqa: F811
    """LN2 of rows of up to 256 values goes half a warp to a row, four rows to a warp: row counts around 4 and 32."""
    x, w = synth.make_tokens(B, N, D, "bf16", seed=41), synth.make_block_weights(D, 4 * D, "bf16", seed=42)
    ref = orc.block_fwd(x.double().numpy(), _np(w), D // 64, 0)
    res = _run_block(ctx, x, w, D // 64, 0, "bf16", torch.float32)
    parity.check_float(res["x_full"].double().numpy(), ref["x_hat"], "bf16", False)


@pytest.mark.parametrize("epilogue", ["bias", "gelu"])
@pytest.mark.parametrize("M,N,K", [(2500, 768, 192), (2500, 768, 384), (9473, 768, 256), (9473, 576, 192), (12700, 576, 64)])
def test_linear_short_k(ctx, M, N, K, epilogue):   # noqa: F811
    """Four (three) groups of epilogue warps: whole tiles, tiles cut in two (two groups idle), a last row tile of a few rows."""
    g = torch.Generator().manual_seed(M + N + K)
    a, w = torch.randn(M, K, generator=g).bfloat16(), (0.1 * torch.randn(N, K, generator=g)).bfloat16()
    b = 0.1 * torch.randn(N, generator=g)
    got = ctx.linear_fwd(a.cuda(), w.cuda(), b.cuda(), epilogue).cpu().double().numpy()
    want = orc.linear(a.double().numpy(), w.double().numpy(), b.double().numpy())
    parity.check_float(got, orc.round_to(orc.gelu(want) if epilogue == "gelu" else want, "bf16"), "bf16", rounded_output=True)


@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual"])
def test_pair_products_back_to_back(ctx, epilogue):   # noqa: F811
    """Pairs with one, two, three and more pieces of work, launch after launch without a pause between them (a CTA's
    shared memory goes to the next launch at once): the same bits every time, and no wait that ran out."""
    g = torch.Generator(device="cuda").manual_seed(9)
    jobs = []
    for M, N, K in [(3000, 768, 320), (9473, 768, 320), (12700, 576, 192), (19200, 768, 320)]:
        a, w = torch.randn(M, K, generator=g, device="cuda").bfloat16(), (0.1 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
        res = torch.randn(M, N, generator=g, device="cuda").bfloat16() if epilogue == "residual" else None
        jobs.append((a, w, res))
    rounds = [[ctx.linear_fwd(a, w, None, epilogue, res) for a, w, res in jobs] for _ in range(25)]
    ctx.async_status()
    for outs in rounds[1:]:
        for first, again in zip(rounds[0], outs):
            assert torch.equal(first, again)
