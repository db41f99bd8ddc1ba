"""The tensor-core products for few rows: row counts around its 128-row tiles, K split over one to eight CTAs, every
epilogue; and the pair-tile kernel's row-mapped residual at a row count that stays with it."""
import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from paper_2508_00367_b200 import synth
from test_gpu_block import _check_block, _np, _run_block, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual"])
@pytest.mark.parametrize("M", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("N,K", [(768, 64), (192, 192), (768, 448), (128, 1536), (768, 768), (2304, 768), (384, 3072)])
def test_linear_few_rows(ctx, M, N, K, epilogue):   # noqa: F811
    g = torch.Generator().manual_seed(M + N + K)
    a, w = torch.randn(M, K, generator=g).bfloat16(), (0.05 * torch.randn(N, K, generator=g)).bfloat16()
    b, res = 0.1 * torch.randn(N, generator=g), torch.randn(M, N, generator=g).bfloat16() if epilogue == "residual" else None
    got = ctx.linear_fwd(a.cuda(), w.cuda(), b.cuda(), epilogue, None if res is None else res.cuda()).cpu().double().numpy()
    want = orc.linear(a.double().numpy(), w.double().numpy(), b.double().numpy())
    if epilogue == "gelu":
        want = orc.gelu(want)
    if epilogue == "residual":
        parity.check_float(got, want + res.double().numpy(), "bf16", rounded_output=False)
    else:
        parity.check_float(got, orc.round_to(want, "bf16"), "bf16", rounded_output=True)


@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual"])
@pytest.mark.parametrize("M,N,K", [(3200, 256, 256), (3201, 256, 256), (6400, 128, 64), (6401, 128, 64), (7040, 256, 128), (7041, 256, 128)])
def test_linear_at_the_lines_of_the_few_row_kernel(ctx, M, N, K, epilogue):   # noqa: F811
    """100 and 220 tiles of 128 x 64: the residual epilogue goes to the pair tiles after the first, the others after the second."""
    g = torch.Generator(device="cuda").manual_seed(M + K)
    a, w = torch.randn(M, K, generator=g, device="cuda").bfloat16(), (0.05 * torch.randn(N, K, generator=g, device="cuda")).bfloat16()
    b, res = 0.1 * torch.randn(N, generator=g, device="cuda"), torch.randn(M, N, generator=g, device="cuda").bfloat16() if epilogue == "residual" else None
    got = ctx.linear_fwd(a, w, b, epilogue, res).cpu().double().numpy()
    want = (a.double() @ w.double().T + b.double()).cpu().numpy()
    if epilogue == "gelu":
        want = orc.gelu(want)
    if epilogue == "residual":
        parity.check_float(got, want + res.cpu().double().numpy(), "bf16", rounded_output=False)
    else:
        parity.check_float(got, orc.round_to(want, "bf16"), "bf16", rounded_output=True)


@pytest.mark.parametrize("mode,dist", [("mlp", "l2"), ("mlp", "cos"), ("mlp_delta", "l1"), ("attn", "l1"), ("attn", "cos"), ("block", "l2")])
def test_block_few_rows_every_score(ctx, mode, dist):   # noqa: F811
    B, N, D, H, r = 1, 130, 384, 6, 40
    x, w = synth.make_tokens(B, N, D, "bf16", seed=11), synth.make_block_weights(D, 4 * D, "bf16", seed=12)
    ref = orc.block_fwd(x.double().numpy(), _np(w), H, r, score_mode=mode, dist=dist)
    res = _run_block(ctx, x, w, H, r, "bf16", torch.float32, score_mode=mode, dist=dist)
    parity.check_float(res["x_full"].double().numpy(), ref["x_hat"], "bf16", False)
    # 5e-4 where the exact x' dominates the distance, else sums of bf16-operand products alone; |m| is a tenth of |x'|
    tol = 5e-4 if (mode, dist) == ("mlp", "l2") else 3e-3 if mode == "mlp_delta" else 2e-3
    rel = np.abs(res["scores"].double().numpy() - ref["scores"]) / np.abs(ref["scores"])
    assert rel.max() < tol, rel.max()


@pytest.mark.parametrize("B,N,D,drops", [(1, 197, 768, [16, 0, 30, 1]), (3, 70, 192, [9, 9, 0]), (16, 197, 384, [16, 30, 0])])
@pytest.mark.parametrize("fold", [False, True])
def test_layer_loop_with_untapped_blocks(ctx, B, N, D, drops, fold):   # noqa: F811
    """Outputs of the last block alone: the loop hands tokens on through row maps (no fold) or with their row sums
    (fold).  Without the fold it must equal the chain of blocks bit for bit; with it every tapped block stays within
    the bf16 tolerance of the oracle fed the loop's own tokens."""
    import paper_2508_00367_b200 as rs
    H = D // 64
    x = synth.make_tokens(B, N, D, "bf16", seed=21).bfloat16().cuda()
    blocks = [synth.make_block_weights(D, 4 * D, "bf16", seed=22 + l) for l in range(len(drops))]
    model = rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, tap_blocks=(), fold_ln1=fold)
    got = model.forward(x)[-1]
    if not fold:
        cur = x
        for l, r in enumerate(drops):
            want = ctx.block_fwd(cur, model.weights[l], H, r)
            cur = want["x_out"]
        torch.cuda.synchronize()
        for k in ("x_out", "scores", "keep_idx"):
            assert torch.equal(got[k], want[k]), k
        return
    cur = x
    for l, o in enumerate(rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, fold_ln1=True).forward(x)):
        ref = orc.block_fwd(cur[:1].double().cpu().numpy(), _np(blocks[l]), H, drops[l])
        s = o["scores"][:1].double().cpu().numpy()
        assert (np.abs(s - ref["scores"]) / ref["scores"]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], o["keep_idx"][:1].cpu().numpy()) == 0:
            parity.check_float(o["x_out"][:1].double().cpu().numpy(), orc.round_to(ref["x_out"], "bf16"), "bf16", True)
        cur = o["x_out"]
    ctx.async_status()


def test_weights_written_just_before_the_block(ctx):   # noqa: F811
    """A product of this library whose output is the next call's weight matrix: the weights that a block requests
    early must be the finished ones."""
    import paper_2508_00367_b200 as rs
    B, N, D = 1, 70, 256
    x = synth.make_tokens(B, N, D, "bf16", seed=31).bfloat16().cuda()
    w = rs.DeviceBlockWeights(synth.make_block_weights(D, 4 * D, "bf16", seed=32), torch.bfloat16, ctx.device)
    eye = torch.eye(D, device="cuda").bfloat16()
    want = ctx.block_fwd(x, w, D // 64, 7)
    torch.cuda.synchronize()
    for name in ("w_qkv", "w_o", "w_fc1"):
        good, wide = w.t[name].clone(), torch.zeros(6000, D, dtype=torch.bfloat16, device="cuda")
        wide[-good.shape[0]:] = good                          # a long product whose last rows are the weights: W I = W
        out = torch.empty_like(wide)
        w.t[name].zero_()
        import ctypes
        setattr(w.struct, name, out.data_ptr() + (6000 - good.shape[0]) * D * 2)
        for _ in range(3):
            out.zero_()
            st = ctx.raw("rs_linear_fwd", 1, 0, 6000, D, D, ctypes.c_void_p(wide.data_ptr()), ctypes.c_void_p(eye.data_ptr()), None, None,
                         ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
            assert st == 0
            got = ctx.block_fwd(x, w, D // 64, 7)
            torch.cuda.synchronize()
            for k in ("x_out", "scores", "keep_idx"):
                assert torch.equal(got[k], want[k]), (name, k)
        w.t[name].copy_(good)
        setattr(w.struct, name, w.t[name].data_ptr())
