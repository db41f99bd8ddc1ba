"""Blocks of 192 columns with more than 512 rows: projection and MLP as one kernel (rs_tail.cuh).  Row counts at the edges of its
tiles of 256 rows and of its rounds, every scored pair and distance, both output types, hidden widths with an odd count of chunks,
the residual through a row map, batches with a count per sample."""
import numpy as np
import pytest
import torch

import parity
from oracle import rs_oracle as orc
from paper_2508_00367_b200 import synth
from test_gpu_block import _check_block, _np, _run_block, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu
D, H = 192, 3


def _launches(ctx, B, N, Dm=4 * D):
    """Kernels of one block call."""
    import paper_2508_00367_b200 as rs
    dw = rs.DeviceBlockWeights(synth.make_block_weights(D, Dm, "bf16", seed=1), torch.bfloat16, ctx.device)
    n = ctx.launch_count()
    ctx.block_fwd(torch.zeros(B, N, D, device="cuda", dtype=torch.bfloat16), dw, H, 1)
    return ctx.launch_count() - n


def test_which_blocks(ctx):   # noqa: F811
    assert _launches(ctx, 2, 256) == 9 and _launches(ctx, 1, 513) == 6 and _launches(ctx, 3, 197) == 6
    assert _launches(ctx, 3, 197, 384) == 6 and _launches(ctx, 3, 197, 576) == 9 and _launches(ctx, 3, 197, 1536) == 9


@pytest.mark.parametrize("out_dtype", [None, torch.float32])
@pytest.mark.parametrize("B,N,Dm", [(1, 513, 768), (2, 320, 384), (3, 256, 128), (1, 769, 768), (5, 127, 768)])
def test_row_counts(ctx, B, N, Dm, out_dtype):   # noqa: F811
    x, w = synth.make_tokens(B, N, D, "bf16", seed=N), synth.make_block_weights(D, Dm, "bf16", seed=Dm)
    res = _run_block(ctx, x, w, H, N // 5, "bf16", out_dtype)
    _check_block(res, orc.block_fwd(x.double().numpy(), _np(w), H, N // 5), "bf16", out_dtype)


@pytest.mark.parametrize("out_dtype", [None, torch.float32])
def test_several_tiles_a_pair(ctx, out_dtype):   # noqa: F811
    """2 x 74 tiles and 148 rows more: a second and a third round; the first and the last samples against the oracle."""
    B, N = (2 * 74 * 256 + 1) // 257 + 1, 257
    x, w = synth.make_tokens(B, N, D, "bf16", seed=7), synth.make_block_weights(D, 4 * D, "bf16", seed=8)
    res = _run_block(ctx, x, w, H, 50, "bf16", out_dtype)
    again = _run_block(ctx, x, w, H, 50, "bf16", out_dtype)
    for k in res:
        assert torch.equal(res[k], again[k]), k
    for b in (0, B // 2, B - 1):
        ref = orc.block_fwd(x[b:b + 1].double().numpy(), _np(w), H, 50)
        _check_block({k: v[b:b + 1] for k, v in res.items()}, ref, "bf16", out_dtype)


def _past_rounds(ctx, rounds):   # noqa: F811
    """(B, N) of the fewest rows above that many whole rounds of 256-row tiles, of samples whose length divides them."""
    first = rounds * (torch.cuda.get_device_properties(ctx.device).multi_processor_count // 2) * 256
    return next((T // N, N) for T in range(first + 1, first + 256) for N in range(128, 63, -1) if T % N == 0)


@pytest.mark.parametrize("mode,dist,out_dtype", [("mlp", "l2", torch.bfloat16), ("attn", "cos", torch.float32), ("block", "l1", torch.bfloat16)])
def test_rows_of_later_rounds(ctx, mode, dist, out_dtype):   # noqa: F811
    """Two whole rounds and a tile of a few rows: bit for bit what the samples give in calls of one round (an eighth of them
    each), where no buffer, barrier or part of tensor memory is used for a second tile."""
    import paper_2508_00367_b200 as rs
    B, N = _past_rounds(ctx, 2)
    x = synth.make_tokens(B, N, D, "bf16", seed=21).bfloat16().cuda()
    dw = rs.DeviceBlockWeights(synth.make_block_weights(D, 4 * D, "bf16", seed=22), torch.bfloat16, ctx.device)
    run = lambda t: ctx.block_fwd(t, dw, H, N // 5, out_dtype=out_dtype, score_mode=mode, dist=dist, want_full=True)   # noqa: E731
    whole, step = run(x), (B + 7) // 8
    assert step * N > 3200                               # (with fewer rows QKV is summed in another order)
    for b in [*range(0, B - step, step), B - step]:
        part = run(x[b:b + step].contiguous())
        for k in part:
            assert torch.equal(whole[k][b:b + step], part[k]), (k, b)
    ctx.async_status()


@pytest.mark.parametrize("mode,dist", [("mlp", "l1"), ("mlp", "cos"), ("mlp_delta", "l2"), ("attn", "l2"), ("attn", "cos"), ("block", "l2"), ("block", "l1")])
def test_scores(ctx, mode, dist):   # noqa: F811
    """Bounds as where these scores come from the epilogues of the single products (bf16 operands in full)."""
    B, N = 3, 190
    x, w = synth.make_tokens(B, N, D, "bf16", seed=51), synth.make_block_weights(D, 4 * D, "bf16", seed=52)
    ref = orc.block_fwd(x.double().numpy(), _np(w), H, 9, score_mode=mode, dist=dist)
    res = _run_block(ctx, x, w, H, 9, "bf16", torch.float32, score_mode=mode, dist=dist)
    parity.check_float(res["x_full"].double().numpy(), ref["x_hat"], "bf16", False)
    err = np.abs(res["scores"].double().numpy() - ref["scores"])
    assert (err if dist == "cos" else err / ref["scores"]).max() < (3e-3 if mode == "mlp_delta" else 2e-3)


@pytest.mark.parametrize("mode", ["mlp", "block"])
def test_rows_through_the_map(ctx, mode):   # noqa: F811
    """The layer loop without dense copies reads the block input through the row map: the bits of chained block calls."""
    import paper_2508_00367_b200 as rs
    B, N, drops = 4, 197, [39, 0, 20, 0]
    x = synth.make_tokens(B, N, D, "bf16", seed=3).bfloat16().cuda()
    blocks = [synth.make_block_weights(D, 4 * D, "bf16", seed=4 + l) for l in range(4)]
    got = rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, tap_blocks=(), score_mode=mode).forward(x)[-1]["x_out"]
    cur = x
    for w, d in zip(blocks, drops):
        cur = ctx.block_fwd(cur, rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device), H, d, score_mode=mode)["x_out"]
    assert torch.equal(got, cur)
    ctx.async_status()


@pytest.mark.parametrize("mode", ["mlp", "block"])
def test_rows_through_the_map_in_later_rounds(ctx, mode):   # noqa: F811
    """The same with two rounds and more behind the map: x of the next tile is copied over the output of the one before."""
    import paper_2508_00367_b200 as rs
    B, N = _past_rounds(ctx, 2)
    x = synth.make_tokens(B, N + 9, D, "bf16", seed=3).bfloat16().cuda()
    blocks, drops = [synth.make_block_weights(D, 4 * D, "bf16", seed=4 + l) for l in range(3)], [9, 0, 8]
    got = rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, tap_blocks=(), score_mode=mode).forward(x)[-1]["x_out"]
    cur = x
    for w, d in zip(blocks, drops):
        cur = ctx.block_fwd(cur, rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device), H, d, score_mode=mode)["x_out"]
    assert torch.equal(got, cur)
    ctx.async_status()


def test_row_sums_in_later_rounds(ctx):   # noqa: F811
    """The folded loop over two rounds and more: every output and score as in loops over an eighth of the samples."""
    import paper_2508_00367_b200 as rs
    B, N = _past_rounds(ctx, 2)
    x = synth.make_tokens(B, N, D, "bf16", seed=13).bfloat16().cuda()
    blocks = [synth.make_block_weights(D, 4 * D, "bf16", seed=14 + l) for l in range(3)]
    run = lambda t: rs.PrunedViT(ctx, blocks, H, [0, 0, 7], torch.bfloat16, fold_ln1=True).forward(t)   # noqa: E731
    whole, step = run(x), (B + 7) // 8
    for b in (0, step, B - step):
        for l, (o, p) in enumerate(zip(whole, run(x[b:b + step].contiguous()))):
            for k in p:
                assert torch.equal(o[k][b:b + step], p[k]), (l, k, b)
    ctx.async_status()


def test_row_sums_for_a_folded_layernorm(ctx):   # noqa: F811
    """Every block of the folded loop against the oracle fed this loop's own input."""
    import paper_2508_00367_b200 as rs
    B, N, drops = 4, 197, [0, 30, 0, 5]
    x = synth.make_tokens(B, N, D, "bf16", seed=13).bfloat16().cuda()
    blocks = [synth.make_block_weights(D, 4 * D, "bf16", seed=14 + l) for l in range(4)]
    outs, cur = rs.PrunedViT(ctx, blocks, H, drops, torch.bfloat16, fold_ln1=True).forward(x), x
    torch.cuda.synchronize()
    for l, o in enumerate(outs):
        ref = orc.block_fwd(cur.double().cpu().numpy(), _np(blocks[l]), H, drops[l])
        s = o["scores"].double().cpu().numpy()
        assert (np.abs(s - ref["scores"]) / ref["scores"]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], o["keep_idx"].cpu().numpy()) == 0:
            parity.check_float(o["x_out"].double().cpu().numpy(), orc.round_to(ref["x_out"], "bf16"), "bf16", True)
        cur = o["x_out"]
    ctx.async_status()


def test_counts_per_sample(ctx):   # noqa: F811
    import paper_2508_00367_b200 as rs
    N, lens = 300, [300, 17, 1, 2, 128, 250, 40]
    drops = [n // 4 for n in lens]
    x = synth.make_tokens(len(lens), N, D, "bf16", seed=11)
    w = synth.make_block_weights(D, 4 * D, "bf16", seed=12)
    dw = rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device)
    dl, dd = (torch.tensor(v, dtype=torch.int32, device="cuda") for v in (lens, drops))
    res = {k: v.cpu() for k, v in ctx.block_fwd_ragged(x.bfloat16().cuda(), dw, H, dl, dd, N).items()}
    for b, n in enumerate(lens):
        ref = orc.block_fwd(x[b:b + 1, :n].double().numpy(), _np(w), H, drops[b])
        s = res["scores"][b, :n].double().numpy()
        assert (np.abs(s - ref["scores"][0]) / ref["scores"][0]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], res["keep_idx"][b:b + 1, :n - drops[b]].numpy()) == 0:
            parity.check_float(res["x_out"][b, :n - drops[b]].double().numpy(), orc.round_to(ref["x_out"][0], "bf16"), "bf16", True)
    ctx.async_status()


def test_counts_with_holes_in_later_rounds(ctx):   # noqa: F811
    """Row tiles of padding in the middle and more tiles in use than two rounds hold: as where nothing is left out, and the oracle."""
    import paper_2508_00367_b200 as rs
    from test_gpu_ragged_skip import _poison
    N, B = 513, 240
    lens = [(N, 1, 1, 400)[b % 4] for b in range(B)]
    starts = [b * N + min(n + 16, N) for b, n in enumerate(lens)]                  # a row tile is in use up to 16 rows past a count
    used = {t for b, e in enumerate(starts) for t in range(b * N // 256, (e - 1) // 256 + 1)}
    assert 148 < len(used) < B * N // 256 <= 1024 and any(t not in used for t in range(20))
    drops = [n // 4 for n in lens]
    x = synth.make_tokens(B, N, D, "bf16", seed=11)
    w = synth.make_block_weights(D, 4 * D, "bf16", seed=12)
    dw = rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device)
    dl, dd = (torch.tensor(v, dtype=torch.int32, device="cuda") for v in (lens, drops))
    xd = x.bfloat16().cuda()
    torch.cuda.empty_cache()
    _poison(1 << 30)
    res = ctx.block_fwd_ragged(xd, dw, H, dl, dd, N)
    full = ctx.block_fwd_ragged(xd, dw, H, dl, dd, N, want_full=True)
    torch.cuda.synchronize()
    assert torch.equal(full["x_out"], res["x_out"]) and torch.equal(full["keep_idx"], res["keep_idx"])
    for b, n in enumerate(lens):
        assert torch.equal(full["scores"][b, :n], res["scores"][b, :n])
    for b in (0, 1, 118, 119, B - 1):
        n, k = lens[b], lens[b] - drops[b]
        ref = orc.block_fwd(x[b:b + 1, :n].double().numpy(), _np(w), H, drops[b])
        s = res["scores"][b, :n].double().cpu().numpy()
        assert (np.abs(s - ref["scores"][0]) / ref["scores"][0]).max() < 5e-4
        if parity.check_keep(ref["scores"], ref["keep_idx"], res["keep_idx"][b:b + 1, :k].cpu().numpy()) == 0:
            parity.check_float(res["x_out"][b, :k].double().cpu().numpy(), orc.round_to(ref["x_out"][0], "bf16"), "bf16", True)
    ctx.async_status()


@pytest.mark.parametrize("Dm", [256, 512, 640])
def test_hidden_widths_without_biases(ctx, Dm):   # noqa: F811
    """The widths between; no biases at all gives what zeros give."""
    B, N = 3, 190
    x, w = synth.make_tokens(B, N, D, "bf16", seed=31), synth.make_block_weights(D, Dm, "bf16", seed=32)
    _check_block(_run_block(ctx, x, w, H, 9, "bf16"), orc.block_fwd(x.double().numpy(), _np(w), H, 9), "bf16", None)
    zero = {k: torch.zeros_like(v) if k.startswith("b_") else v for k, v in w.items()}
    none = {k: None if k.startswith("b_") else v for k, v in w.items()}
    res, bare = (_run_block(ctx, x, v, H, 9, "bf16") for v in (zero, none))
    _check_block(bare, orc.block_fwd(x.double().numpy(), _np(zero), H, 9), "bf16", None)
    for k in res:
        assert torch.equal(res[k], bare[k]), k


@pytest.mark.parametrize("mode,dist", [("mlp", "l2"), ("attn", "cos"), ("block", "l1")])
def test_rows_that_are_not_finite(ctx, mode, dist):   # noqa: F811
    """Infinities and NaN in one sample make all of that sample NaN (its keys are) and no bit of the others, in the same tiles."""
    B, N = 20, 60
    x, w = synth.make_tokens(B, N, D, "bf16", seed=41), synth.make_block_weights(D, 4 * D, "bf16", seed=42)
    clean = _run_block(ctx, x, w, H, 0, "bf16", torch.float32, score_mode=mode, dist=dist)
    bad = {3: float("inf"), 4: -float("inf"), 11: float("nan")}
    for b, v in bad.items():
        x[b, 7 * (b % 3), 5] = v
    res = _run_block(ctx, x, w, H, 0, "bf16", torch.float32, score_mode=mode, dist=dist)
    for b in range(B):
        for k in ("x_full", "scores"):
            assert torch.isnan(res[k][b]).all() if b in bad else torch.equal(res[k][b], clean[k][b]), (k, b)
    ctx.async_status()
