"""Measured cases: what a program that uses this library has it do, through the public entry points.

A case is a dict of plain values; `kind` names the entry point:

  vit     PrunedViT.forward: the whole pruned forward pass (LN1 folded, as bench.py runs it)
  ragged  Context.vit_fwd_ragged: the forward pass on a padded batch with a token count per sample
  block   Context.block_fwd: one block, its score and its pruning
  attn    Context.attn_fwd on a packed [B, N, 3, H, 64] projection
  prune   Context.shift_score, then Context.topk_compact on the tokens it scored
  lines   Context.shift_score, then Context.linewise_compact on a feature map

Tokens come in bands of magnitude, one band per pruning step (the tokens a step removes are the weakest
band left, in random places), with distances between the bands that rounding cannot bridge: which
tokens are kept then depends on the inputs and not on the order of a sum, so outputs can be compared
row by row.  Weights are N(0, 0.02) as in the repository's synthetic workloads; video tokens are
correlated from frame to frame (AR(1), 0.9) as there.
"""
import math

import numpy as np
import torch

import paper_2508_00367_b200 as rs
from paper_2508_00367_b200.synth import WORKLOADS

DT = {"f32": torch.float32, "bf16": torch.bfloat16}
# the largest listed case is video_vit_l14; drawn cases stay below its arithmetic and below this much memory traffic
FLOPS_MAX = 7.5e12
TOKENS_MAX = 120_000


# ------------------------------------------------------------------ schedules

def drops_of(case):
    """Tokens removed after each block (host schedule of a `vit` or `ragged` case at its full length)."""
    if case.get("workload"):
        return list(WORKLOADS[case["workload"]].drops)
    n, out = case["N"], []
    at = [int(a) for a in str(case["at"]).split(",")] if case["at"] != "all" else None
    for l in range(1, case["L"] + 1):
        d = 0
        if at is None or l in at:
            d = int(case["r"]) if case["r"] >= 1 else int(math.floor(case["r"] * n))
        d = max(0, min(d, n - 1))
        out.append(d)
        n -= d
    return out


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # One ViT-S block in fp32, two images: the smallest call, the precision of a reference run.
        dict(name="block_vit_s_f32", kind="block", dtype="f32", out="f32", B=2, N=197, D=384, r=16, mode="mlp", dist="l2"),
        # One block on a mid-sized batch with another operation choice and fp32 outputs (what a study of the
        # scores calls, block by block).
        dict(name="block_vit_l_attn_score", kind="block", dtype="bf16", out="f32", B=8, N=577, D=1024, r=115, mode="attn", dist="l2"),
        # One image through ViT-B/16 as a server answers it: a captured graph over a fixed input buffer.
        dict(name="vit_b16_one_image", kind="vit", graph=True, B=1, N=197, D=768, L=12, r=16, at="all", frames=0),
        # DeiT-T as the paper prunes it (20 % after blocks 1, 4 and 7), half the paper's batch: three heads.
        dict(name="deit_t_batch", kind="vit", graph=False, B=256, N=197, D=192, L=12, r=0.2, at="1,4,7", frames=0),
        # The four bf16 workloads of the repository, from images to long clips, by the plain call.
        dict(name="vit_b16", kind="vit", graph=False, workload="vit_b16", B=64, N=197, D=768, L=12, frames=0),
        dict(name="vit_l16_384", kind="vit", graph=False, workload="vit_l16_384", B=32, N=577, D=1024, L=24, frames=0),
        dict(name="video_vit_b16", kind="vit", graph=False, workload="video_vit_b16", B=16, N=1569, D=768, L=12, frames=8),
        dict(name="video_vit_l14", kind="vit", graph=False, workload="video_vit_l14", B=4, N=4097, D=1024, L=24, frames=16),
        # Clips of different lengths in one padded batch, a ratio of each clip's own tokens dropped.
        dict(name="ragged_clips", kind="ragged", B=12, N=1177, D=768, L=12, r=0.2, at="1,4,7", shortest=0.25),
        # The attention entry point alone, a clip with an odd number of tokens.
        dict(name="attn_clip", kind="attn", dtype="bf16", B=2, N=2353, H=12),
        # Score and compaction as a pass of their own between two sub-layers of somebody else's model.
        dict(name="prune_images", kind="prune", dtype="bf16", dist="l2", B=512, N=197, D=768, r=16),
        # A ResNet-50 first-stage feature map pruned line by line.
        dict(name="lines_resnet50", kind="lines", dtype="bf16", B=64, H=56, W=56, C=256, dr=8, dc=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vit_flops(B, counts, D):
    return sum(24.0 * B * n * D * D + 4.0 * B * n * n * D for n in counts)


def draw(rng):
    kind = rng.choice(["vit", "vit", "vit", "vit", "ragged", "block", "block", "attn", "prune", "lines"])
    if kind in ("vit", "ragged"):
        while True:
            # (batches with a count per sample need widths of 128)
            D, L = rng.choice(([192] if kind == "vit" else []) + [384, 768, 768, 1024, 1024]), rng.choice([6, 12, 12, 24])
            N, frames = _log(rng, 65, 2353), 0
            if kind == "vit" and rng.random() < 0.4:
                frames = rng.choice([4, 8, 12, 16])
                N = 1 + frames * _log(rng, 49, 256)
            at, r = rng.choice([("all", max(1, N // (L + 2))), ("1,4,7", 0.2), ("1,2,3", 0.2), ("3,6,9", 0.3), ("1,2,3", 0.1)])
            if L == 6 and at == "3,6,9":
                continue
            case = dict(kind=kind, B=1, N=N, D=D, L=L, r=r, at=at)
            counts = _counts(N, drops_of(case))
            most = int(min(256, FLOPS_MAX / _vit_flops(1, counts, D), TOKENS_MAX / N))
            if most < 1:
                continue
            case["B"] = _log(rng, 1, most)
            if kind == "ragged":
                case["shortest"] = round(rng.uniform(0.1, 0.9), 2)
                case["at"], case["r"] = (at, r) if at != "all" else ("1,4,7", 0.2)
            else:
                case.update(frames=frames, graph=case["B"] * N < 2500)
            return case
    if kind == "block":
        dtype = rng.choice(["f32", "bf16", "bf16"])
        D = rng.choice([192, 384, 768, 1024])
        N = _log(rng, 50, 577 if dtype == "f32" else 4097)
        B = _log(rng, 1, max(1, min(128, (12_000 if dtype == "f32" else 60_000) // N)))
        mode, dist = rng.choice([("mlp", "l2"), ("mlp", "l2"), ("mlp", "l1"), ("attn", "l2"), ("attn", "l1")])
        out = "f32" if dtype == "f32" else rng.choice(["bf16", "bf16", "f32"])
        return dict(kind=kind, dtype=dtype, out=out, B=B, N=N, D=D, r=max(1, int(N * rng.choice([0.08, 0.2, 0.3]))), mode=mode, dist=dist)
    if kind == "attn":
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        H, N = rng.choice([3, 6, 12, 16]), _log(rng, 17, 4608 if dtype == "bf16" else 800)
        return dict(kind=kind, dtype=dtype, B=_log(rng, 1, max(1, min(256, TOKENS_MAX // N, int((3e11 if dtype == "bf16" else 2e10) / (256.0 * N * N * H))))), N=N, H=H)
    if kind == "prune":
        dtype, D = rng.choice(["bf16", "bf16", "f32"]), rng.choice([192, 384, 768, 1024])
        N = _log(rng, 50, 16384)
        B = _log(rng, 1, max(1, min(512, int(160e6 / (N * D)))))
        return dict(kind=kind, dtype=dtype, dist=rng.choice(["l2", "l2", "l1", "cos"]), B=B, N=N, D=D, r=max(1, int(N * rng.choice([0.08, 0.2, 0.3, 0.5]))))
    side, C = rng.choice([(56, 64), (56, 256), (28, 512), (28, 128), (14, 1024), (63, 256)])
    H, W = side, max(4, side - rng.choice([0, 0, 3, 7]))
    return dict(kind=kind, dtype=rng.choice(["bf16", "bf16", "f32"]), B=_log(rng, 1, max(1, int(60e6 / (H * W * C)))), H=H, W=W, C=C,
                dr=max(1, H // rng.choice([4, 7, 14])), dc=max(1, W // rng.choice([4, 7, 14])))


# ------------------------------------------------------------------ inputs

def _counts(n, drops):
    out = []
    for d in drops:
        out.append(n)
        n -= d
    return out


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _weights(g, D, Dm, dtype):
    mat = lambda *s: (0.02 * _randn(g, *s)).to(dtype)           # noqa: E731
    vec = lambda n, base=0.0: (base + 0.02 * _randn(g, n))      # noqa: E731
    return dict(w_qkv=mat(3 * D, D), w_o=mat(D, D), w_fc1=mat(Dm, D), w_fc2=mat(D, Dm), b_qkv=vec(3 * D), b_o=vec(D), b_fc1=vec(Dm),
                b_fc2=vec(D), ln1_g=vec(D, 1.0), ln1_b=vec(D), ln2_g=vec(D, 1.0), ln2_b=vec(D))


def _bands(g, B, N, steps, lens=None):
    """[B, N] band numbers: of every sample's tokens, steps[k][b] random ones in band k, the rest (and token 0) on top."""
    key = torch.rand(B, N, generator=g, device="cuda")
    key[:, 0] = 2.0
    if lens is not None:
        key = torch.where(torch.arange(N, device="cuda")[None] < lens[:, None], key, torch.full_like(key, 3.0))
    rank = key.argsort(dim=1).argsort(dim=1)
    band, cut = torch.zeros_like(rank), torch.zeros(B, dtype=torch.long, device="cuda")
    for s in steps:
        cut = cut + torch.as_tensor(s, device="cuda")
        band += rank >= cut[:, None]
    return band


def _tokens(g, B, N, D, band, n_steps, frames=0):
    """Unit-rms tokens times the magnitude of their band."""
    if frames:
        P = (N - 1) // frames
        x = torch.empty(B, N, D, device="cuda")
        x[:, 0] = _randn(g, B, D)
        f = x[:, 1:].view(B, frames, P, D)
        f[:, 0] = _randn(g, B, P, D)
        for t in range(1, frames):
            f[:, t] = 0.9 * f[:, t - 1] + math.sqrt(1.0 - 0.81) * _randn(g, B, P, D)
    else:
        x = _randn(g, B, N, D)
    x = x / x.square().mean(dim=2, keepdim=True).sqrt()
    return x * (_band_step(n_steps) ** band)[:, :, None]


def _band_step(n_steps):
    return 1.5 if n_steps <= 4 else 1.25 if n_steps <= 12 else 1.17


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    ctx = rs.Context(0)
    s = dict(case=case, ctx=ctx)
    if kind in ("vit", "ragged"):
        B, N, D, L = case["B"], case["N"], case["D"], case["L"]
        drops = drops_of(case)
        blocks = [_weights(g, D, 4 * D, torch.bfloat16) for _ in range(L)]
        if kind == "vit":
            steps = [d for d in drops if d]
            s["x"] = _tokens(g, B, N, D, _bands(g, B, N, steps), len(steps), case["frames"]).to(torch.bfloat16)
            model = rs.PrunedViT(ctx, blocks, D // 64, drops, torch.bfloat16, tap_blocks=(), fold_ln1=True)
            model.plan(B, N, D)
            s["model"] = model
            if case["graph"]:
                s["slot"] = torch.empty_like(s["x"])
                model.forward(s["slot"].zero_(), graph=True)
        else:
            lens = np.random.RandomState(seed % (1 << 31)).randint(max(2, int(case["shortest"] * N)), N + 1, B)
            lens[0] = N
            n, per, pad, width = lens.copy(), [], [], N
            for l, d in enumerate(drops):
                own = np.floor(case["r"] * n).astype(np.int64) if d else np.zeros_like(n)
                own = np.minimum(own, n - 1)
                n = n - own
                per.append(own)
                pad.append(int(width - n.max()))
                width = int(n.max())
            dl = torch.as_tensor(lens, device="cuda")
            steps = [p for p in per if p.any()]
            x = _tokens(g, B, N, D, _bands(g, B, N, steps, dl), len(steps))
            x[torch.arange(N, device="cuda")[None] >= dl[:, None]] = 0.0
            s.update(x=x.to(torch.bfloat16), weights=[rs.DeviceBlockWeights(w, torch.bfloat16, ctx.device) for w in blocks], pad=pad,
                     lens=dl.to(torch.int32), drops=torch.as_tensor(np.stack(per), device="cuda").to(torch.int32))
    elif kind == "block":
        B, N, D, dt = case["B"], case["N"], case["D"], DT[case["dtype"]]
        s["x"] = _tokens(g, B, N, D, _bands(g, B, N, [case["r"]]), 1).to(dt)
        s["weights"] = rs.DeviceBlockWeights(_weights(g, D, 4 * D, dt), dt, ctx.device)
    elif kind == "attn":
        qkv = _randn(g, case["B"], case["N"], 3, case["H"], 64).to(DT[case["dtype"]])
        s.update(q=qkv[:, :, 0], k=qkv[:, :, 1], v=qkv[:, :, 2])
    elif kind == "prune":
        B, N, D, dt = case["B"], case["N"], case["D"], DT[case["dtype"]]
        s["before"] = _randn(g, B, N, D).to(dt)
        shift = 0.1 * torch.pow(2.0, _bands(g, B, N, [case["r"]]).float())          # the kept tokens moved twice as far
        s["after"] = (s["before"].float() + shift[:, :, None] * _randn(g, B, N, D)).to(dt)
    else:
        B, H, W, C, dt = case["B"], case["H"], case["W"], case["C"], DT[case["dtype"]]
        s["before"] = _randn(g, B, H * W, C).to(dt)
        shift = 0.1 * (_bands(g, B, H, [case["dr"]]).float()[:, :, None] + _bands(g, B, W, [case["dc"]]).float()[:, None, :] + 0.5)
        s["after"] = (s["before"].float() + shift.view(B, H * W, 1) * _randn(g, B, H * W, C)).to(dt)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "vit":
        if case["graph"]:
            s["slot"].copy_(s["x"])
            return s["model"].forward(s["slot"], graph=True)
        return s["model"].forward(s["x"])
    if kind == "ragged":
        return ctx.vit_fwd_ragged(s["x"], s["weights"], case["D"] // 64, s["pad"], s["lens"], s["drops"])
    if kind == "block":
        return ctx.block_fwd(s["x"], s["weights"], case["D"] // 64, case["r"], out_dtype=DT[case["out"]], score_mode=case["mode"], dist=case["dist"])
    if kind == "attn":
        return ctx.attn_fwd(s["q"], s["k"], s["v"])
    scores = ctx.shift_score(s["after"], s["before"], dist=case.get("dist", "l2"))
    if kind == "prune":
        x_out, keep = ctx.topk_compact(scores, s["after"], case["r"])
        return dict(scores=scores, x_out=x_out, keep_idx=keep)
    B, H, W, C = case["B"], case["H"], case["W"], case["C"]
    x_out, rows, cols = ctx.linewise_compact(scores.view(B, H, W), s["after"].view(B, H, W, C), case["dr"], case["dc"])
    return dict(scores=scores, x_out=x_out, keep_rows=rows, keep_cols=cols)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind = case["kind"]
    sz = 2 if case.get("dtype", "bf16") == "bf16" else 4
    if kind in ("vit", "ragged"):
        B, N, D, L = case["B"], case["N"], case["D"], case["L"]
        drops = drops_of(case)
        counts = _counts(N, drops)
        weights = L * (12 * D * D * 2 + 13 * D * 4 + 4 * D)
        n_out = N - sum(drops)
        if kind == "vit":
            lists = sum(B * (n + n - d) * 4 for n, d in zip(counts, drops) if d)
            return dict(bytes=weights + B * (N + n_out) * D * 2 + lists, flops=_vit_flops(B, counts, D))
        # lengths are uniform between the shortest and the longest sample: their mean, and the mean of their squares
        a = case["shortest"]
        m1, m2 = (1 + a) / 2, (1 + a + a * a) / 3
        flops = sum(24.0 * B * n * m1 * D * D + 4.0 * B * n * n * m2 * D for n in counts)
        return dict(bytes=weights + B * m1 * N * D * 2 + B * n_out * (D * 2 + 4), flops=flops)
    if kind == "block":
        B, N, D, K = case["B"], case["N"], case["D"], case["N"] - case["r"]
        osz = 2 if case["out"] == "bf16" else 4
        return dict(bytes=12 * D * D * sz + 13 * D * 4 + B * N * D * sz + B * K * D * osz + B * (N + K) * 4, flops=_vit_flops(B, [N], D))
    if kind == "attn":
        B, N, D = case["B"], case["N"], case["H"] * 64
        return dict(bytes=4 * B * N * D * sz, flops=4.0 * B * N * N * D)
    if kind == "prune":
        B, N, D, K = case["B"], case["N"], case["D"], case["N"] - case["r"]
        # both inputs for the score, then the kept rows out (the rows were read for the score already)
        return dict(bytes=2 * B * N * D * sz + B * K * D * sz + B * (N + K) * 4, flops=3.0 * B * N * D)
    B, H, W, C = case["B"], case["H"], case["W"], case["C"]
    K = (H - case["dr"]) * (W - case["dc"])
    return dict(bytes=2 * B * H * W * C * sz + B * K * C * sz + B * H * W * 4 + B * (H - case["dr"] + W - case["dc"]) * 4, flops=3.0 * B * H * W * C)


def tolerance(case):
    """Relative errors (2-norm), about four times what was seen: fp32 entry points against the same arithmetic in 64 bits;
    bf16 ones against themselves with the other attention kernel and with the fp32-FMA kernels (other tiles, other sums)."""
    kind = case["kind"]
    if kind in ("prune", "lines"):
        # sums of up to 1024 products in fp32 (seen 5e-8); 1 - cos of nearly parallel rows cancels (seen 4e-6)
        return dict(rel=2e-5 if case.get("dist") == "cos" else 1e-6)
    if case.get("dtype") == "f32":
        return dict(rel=3e-6)              # seen 7e-7
    if kind == "attn":
        return dict(rel=1e-2)              # P rounded to bf16, bf16 output: seen 2.5e-3
    if kind == "block":
        return dict(rel=4e-3)              # seen 1e-3
    return dict(rel=2.5e-2)                # up to 24 blocks, each rounding the residual stream to bf16: seen 6e-3
