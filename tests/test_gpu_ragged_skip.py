"""Row tiles of padding are left out of the products and LayerNorms of a batch with a count per sample: whatever the
buffers held there before (NaN here) must not reach a row in use."""
import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from paper_2508_00367_b200 import synth
from test_gpu_block import _np, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


def _poison(nbytes=1 << 28):
    t = torch.full((nbytes // 4,), float("nan"), device="cuda")      # the caching allocator hands this memory out next
    torch.cuda.synchronize()
    del t


@pytest.mark.parametrize("lens", [[300, 1, 17, 128, 250, 2, 40, 129, 113], [300, 300, 1, 1, 1, 1, 1, 1, 300], [3] * 8 + [300]])
@pytest.mark.parametrize("N,D", [(300, 384), (1100, 256), (1100, 192)])
def test_block_over_poisoned_buffers(ctx, lens, N, D):   # noqa: F811
    import paper_2508_00367_b200 as rs
    B, H = 9, D // 64
    lens = [min(n if n != 300 else N, N) for n in lens]
    drops = [n // 4 for n in lens]
    x = synth.make_tokens(B, N, D, "bf16", seed=N)
    for b, n in enumerate(lens):
        x[b, n:] = 0
    w = synth.make_block_weights(D, 4 * D, "bf16", seed=N + 1)
    dw = rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device)
    dl, dd = (torch.tensor(v, dtype=torch.int32, device="cuda") for v in (lens, drops))
    xd = x.bfloat16().cuda()
    torch.cuda.empty_cache()
    _poison()
    res = ctx.block_fwd_ragged(xd, dw, H, dl, dd, N)
    torch.cuda.synchronize()
    res = {k: v.cpu() for k, v in res.items()}
    assert torch.isfinite(res["scores"]).all() and torch.isfinite(res["x_out"].float()).all()
    for b in (0, 1, 2, 7, 8):
        n, k = lens[b], lens[b] - drops[b]
        ref = orc.block_fwd(x[b:b + 1, :n].double().numpy(), _np(w), H, drops[b])
        s = res["scores"][b, :n].double().numpy()
        assert (np.abs(s - ref["scores"][0]) / ref["scores"][0]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], res["keep_idx"][b:b + 1, :k].numpy()) == 0:
            parity.check_float(res["x_out"][b, :k].double().numpy(), orc.round_to(ref["x_out"][0], "bf16"), "bf16", True)
        assert (res["x_out"][b, k:] == 0).all() and (res["keep_idx"][b, k:] == -1).all()
    # with the un-pruned output asked for nothing is left out: the same rows, and finite ones in the padding
    torch.cuda.empty_cache()
    _poison()
    full = ctx.block_fwd_ragged(xd, dw, H, dl, dd, N, want_full=True)
    torch.cuda.synchronize()
    assert torch.equal(full["x_out"].cpu(), res["x_out"])
    assert torch.isfinite(full["x_full"].float()).all() and torch.isfinite(full["scores"]).all()
    ctx.async_status()


@pytest.mark.parametrize("D", [192, 256, 384])                        # LN2 in the kernel for 192 columns, both LayerNorm kernels
@pytest.mark.parametrize("counts", [[2147483647, 2147483640, 1300, 40], [0, -5, -2147483648, 300]])
def test_counts_outside_the_sample_are_clamped(ctx, counts, D):   # noqa: F811
    """seq_lens holds any int: it stands for its value clamped to [1, N], in every kernel, over poisoned buffers too."""
    import paper_2508_00367_b200 as rs
    N, B = 300, 4
    x = synth.make_tokens(B, N, D, "bf16", seed=5).bfloat16().cuda()
    dw = rs.DeviceBlockWeights(synth.make_block_weights(D, 4 * D, "bf16", seed=6), torch.bfloat16, ctx.device)
    drops = torch.tensor([0, 30, 0, 7], dtype=torch.int32, device="cuda")
    got = []
    for c in (counts, [min(max(n, 1), N) for n in counts]):
        dl = torch.tensor(c, dtype=torch.int32, device="cuda")
        torch.cuda.empty_cache()
        _poison()
        res = ctx.block_fwd_ragged(x, dw, D // 64, dl, drops, N)
        torch.cuda.synchronize()
        got.append({k: v.cpu() for k, v in res.items()})
    assert torch.isfinite(got[0]["scores"]).all() and torch.isfinite(got[0]["x_out"].float()).all()
    for k in got[0]:
        assert torch.equal(got[0][k], got[1][k]), k
    ctx.async_status()
