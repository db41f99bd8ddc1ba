"""Selection and row gather at the edges of their launch rules: keys per thread change after 1024, 2048, 5120 and
16384 tokens; rows of up to 32 and 64 sixteen-byte pieces are moved several to a warp."""
import numpy as np
import pytest
import torch

from oracle import rs_oracle as orc
from test_gpu_parts import _scores, ctx   # noqa: F401  (the module's context fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["normal", "ties", "special", "equal"])
@pytest.mark.parametrize("N", [2048, 2049, 5120, 5121, 16384, 16385])
def test_selection_at_the_keys_per_thread_edges(ctx, kind, N):   # noqa: F811
    s = _scores(2, N, kind, N)
    for has_cls in (True, False):
        for r in (1, N // 3, N - 2, N - 1):
            _, keep = ctx.topk_compact(torch.from_numpy(s).cuda(), None, r, has_cls)
            np.testing.assert_array_equal(keep.cpu().numpy(), orc.topk(s.astype(np.float64), r, has_cls), err_msg=f"r={r} cls={has_cls}")


@pytest.mark.parametrize("pieces", [1, 31, 32, 33, 63, 64, 65, 300])
@pytest.mark.parametrize("B,N,r", [(1, 3, 1), (3, 50, 7)])       # row counts that leave a warp partly filled
def test_rows_of_every_width_class(ctx, pieces, B, N, r):   # noqa: F811
    D = 8 * pieces
    s = _scores(B, N, "normal", pieces)
    x = torch.randn(B, N, D, generator=torch.Generator().manual_seed(pieces)).bfloat16()
    buf = torch.full((B * (N - r) * D + 128,), -7.0, dtype=torch.bfloat16, device="cuda")      # canaries around the rows
    xo = buf[64:-64].view(B, N - r, D)
    _, keep = ctx.topk_compact(torch.from_numpy(s).cuda(), x.cuda(), r, True, x_out=xo)
    want = orc.topk(s.astype(np.float64), r, True)
    np.testing.assert_array_equal(keep.cpu().numpy(), want)
    assert torch.equal(xo.cpu(), torch.stack([x[b][torch.from_numpy(want[b]).long()] for b in range(B)]))
    assert (buf[:64] == -7).all() and (buf[-64:] == -7).all()
