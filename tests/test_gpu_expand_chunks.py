"""The expansion at the edges of its 256-pixel chunks, of its blocks and of the median's blocks (2048 pixels), with the
arrays full in the middle of a chunk: the mask, the ranks and the copied rows are exact (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [0, 4, 16])
@pytest.mark.parametrize("sizes", [[(1, 1)], [(255, 1)], [(16, 16)], [(257, 1)], [(89, 23)], [(64, 32)], [(683, 3)],
                                   [(33, 31), (1, 7), (70, 59)]])
def test_chunk_edges(sizes, d):
    cams = [synth.camera(w, h, 50.0) for w, h in sizes]
    r = raster.Renderer(5, cams, d, 64)
    rng = np.random.default_rng(sum(w * h for w, h in sizes) + d)
    P = r.P
    sil, dgt = rng.random(P, np.float32), (rng.random(P, np.float32) + 1) * (rng.random(P) < 0.9)
    e = np.where(rng.random(P) < 0.1, 1.0, 2.0 ** -8).astype(np.float32) * rng.random(P, np.float32)
    dgt = dgt.astype(np.float32)
    depth = dgt + e
    rgb = rng.random((3, P), np.float32)
    up = lambda x: torch.as_tensor(x).cuda()
    for buf, x in ((r.img_sil, sil), (r.img_depth, depth)):
        buf.copy_(up(x))
    f = raster.Field(*(torch.randn(s, device="cuda") for s in ((5, 3), (5, 4), (5, 3), (5,), (5, 3), (5, d))))
    tg = dict(rgb=up(rgb), depth=up(dgt), label=torch.zeros(P, dtype=torch.uint8, device="cuda"))
    mask = np.zeros(P, bool)
    for v in range(len(sizes)):
        s = slice(r.pix_off[v], r.pix_off[v + 1])
        err = np.abs(depth[s] - dgt[s])
        seen = dgt[s] > 0
        med = np.float32(oracle.lower_median(err[seen].astype(np.float64))) if seen.any() else np.float32(0)
        mask[s] = seen & ((sil[s] < 0.5) | ((depth[s] > dgt[s]) & (err > np.float32(50) * med)))
    want = np.flatnonzero(mask)
    for room in {max(x, 1) for x in (P, len(want), len(want) - 3, len(want) // 2)}:  # no room is refused
        feat = torch.randn(room, d, device="cuda")
        out, src, total, status = raster.expand(r, f, tg, feat)
        k = min(room, len(want))
        assert total == len(want) and out.n == 5 + k and status == (L.GS_ERR_CAPACITY if k < total else 0)
        np.testing.assert_array_equal(src.cpu().numpy(), want[:k])
        assert torch.equal(out.means[:5], f.means) and torch.equal(out.feat, torch.cat([f.feat, feat[:k]]))
        np.testing.assert_array_equal(out.rgb[5:].cpu().numpy(), rgb[:, want[:k]].T)
