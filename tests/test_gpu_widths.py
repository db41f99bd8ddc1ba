"""Output widths of the tensor-core products that are whole tiles of 192 but not of 128 columns (D = 192: three heads)."""
import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from paper_2508_00367_b200 import synth
from test_gpu_block import _check_block, _np, _run_block, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("epilogue", ["bias", "gelu", "residual"])
@pytest.mark.parametrize("M,N,K", [(77, 192, 192), (300, 576, 192), (257, 960, 64), (1, 192, 768)])
def test_linear_widths_of_192(ctx, epilogue, M, N, K):   # noqa: F811
    g = torch.Generator().manual_seed(M + N)
    a, w = torch.randn(M, K, generator=g).bfloat16(), (0.05 * torch.randn(N, K, generator=g)).bfloat16()
    b, res = 0.1 * torch.randn(N, generator=g), torch.randn(M, N, generator=g).bfloat16() if epilogue == "residual" else None
    assert ctx.linear_uses_tensor_cores(torch.bfloat16, M, N, K)
    got = ctx.linear_fwd(a.cuda(), w.cuda(), b.cuda(), epilogue, None if res is None else res.cuda()).cpu().double().numpy()
    want = orc.linear(a.double().numpy(), w.double().numpy(), b.double().numpy())
    if epilogue == "gelu":
        want = orc.gelu(want)
    if epilogue == "residual":
        parity.check_float(got, want + res.double().numpy(), "bf16", rounded_output=False)
    else:
        parity.check_float(got, orc.round_to(want, "bf16"), "bf16", rounded_output=True)


@pytest.mark.parametrize("out_dtype", [None, torch.float32])
def test_block_of_three_heads(ctx, out_dtype):   # noqa: F811
    B, N, D, H, r = 3, 197, 192, 3, 39
    x, w = synth.make_tokens(B, N, D, "bf16", seed=1), synth.make_block_weights(D, 4 * D, "bf16", seed=2)
    desc = ctx.block_desc(B, N, D, H, 4 * D, r, torch.bfloat16)
    assert ctx.block_uses_tensor_cores(desc)
    res = _run_block(ctx, x, w, H, r, "bf16", out_dtype)
    _check_block(res, orc.block_fwd(x.double().numpy(), _np(w), H, r), "bf16", out_dtype)


def test_layer_loop_of_three_heads_with_folded_ln1(ctx):   # noqa: F811
    """The folded loop at D = 192: every block against the oracle fed this loop's own input."""
    import paper_2508_00367_b200 as rs
    B, N, D, H, drops = 2, 197, 192, 3, [39, 0, 31]
    x = synth.make_tokens(B, N, D, "bf16", seed=3).bfloat16().cuda()
    blocks = [synth.make_block_weights(D, 4 * D, "bf16", seed=4 + l) for l in range(3)]
    model = rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, fold_ln1=True)
    assert "w_qkv_ln" in model.weights[1].t
    outs, cur = model.forward(x), x
    torch.cuda.synchronize()
    for l, o in enumerate(outs):
        ref = orc.block_fwd(cur.double().cpu().numpy(), _np(blocks[l]), H, drops[l])
        s = o["scores"].double().cpu().numpy()
        assert (np.abs(s - ref["scores"]) / ref["scores"]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], o["keep_idx"].cpu().numpy()) == 0:
            parity.check_float(o["x_out"].double().cpu().numpy(), orc.round_to(ref["x_out"], "bf16"), "bf16", True)
        cur = o["x_out"]
    ctx.async_status()


@pytest.mark.parametrize("B,N,D", [(4, 50, 192), (3, 1, 192), (2, 64, 192), (31, 100, 192), (60, 128, 192), (2, 129, 192), (32, 197, 192), (1, 65, 576),
                                   (3, 320, 576), (2, 513, 960), (1, 1201, 192)])
def test_attention_weights_of_these_widths(ctx, B, N, D, monkeypatch):   # noqa: F811
    """These blocks ran on the fp32-FMA kernels with fp32 attention weights: the error of what attention adds, against 64
    bits, stays what those kernels make of the same roundings (bf16 weights: 1.04 to 1.19 times as much)."""
    import paper_2508_00367_b200 as rs
    monkeypatch.setenv("RS_DISABLE_TC", "1")
    fma = rs.Context(0)
    monkeypatch.delenv("RS_DISABLE_TC")
    x, w = synth.make_tokens(B, N, D, "bf16", seed=N), synth.make_block_weights(D, 4 * D, "bf16", seed=D)
    # values well above the other terms' roundings: attention's output counts
    w["w_qkv"][2 * D:] *= 8
    wd = {k: v.double().cuda() for k, v in w.items()}
    xd = x.double().cuda()
    u = torch.nn.functional.layer_norm(xd, (D,), wd["ln1_g"], wd["ln1_b"], 1e-6)
    q, k, v = (u @ wd["w_qkv"].T + wd["b_qkv"]).view(B, N, 3, D // 64, 64).permute(2, 0, 3, 1, 4)
    att = (torch.softmax(q @ k.transpose(2, 3) / 8.0, -1) @ v).transpose(1, 2).reshape(B, N, D)
    want = (att @ wd["w_o"].T + wd["b_o"]).norm(dim=-1)
    err = []
    for c in (ctx, fma):
        dw = rs.DeviceBlockWeights(w, torch.bfloat16, c.device)
        res = c.block_fwd(x.bfloat16().cuda(), dw, D // 64, 0, out_dtype=torch.float32, score_mode="attn")
        c.async_status()
        err.append((res["scores"].double() - ((att @ wd["w_o"].T + wd["b_o"]) - xd).norm(dim=-1)).norm().item())
    assert want.min() > 0 and err[0] <= 1.02 * err[1], err
    fma.close()
