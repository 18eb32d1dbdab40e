"""The SSIM term at the edges of its 32x32 tiles and 11x11 window, over views of different sizes, against the oracle, and
the exactness of its sum (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu

ONLY_SSIM = raster.LossWeights(color=1.0, depth=0.0, sem=0.0, big=0.0, small=0.0, ssim=1.0)


def _ssim_loss(imgs, tgts):
    """The renderer after a loss of the SSIM term alone on [3, H, W] f32 images."""
    r = raster.Renderer(0, [synth.camera(x.shape[2], x.shape[1], 60.0) for x in imgs], 0, 0)
    flat = lambda xs: torch.as_tensor(np.concatenate([x.reshape(3, -1) for x in xs], 1)).cuda()
    r.img_rgb.copy_(flat(imgs))
    tg = dict(rgb=flat(tgts), depth=torch.zeros(r.P, device="cuda"),
              label=torch.full((r.P,), 255, dtype=torch.uint8, device="cuda"))
    r.loss(tg, None, None, ONLY_SSIM)
    return r


@pytest.mark.parametrize("sizes", [[(1, 1)], [(5, 7)], [(11, 3)], [(31, 33)], [(32, 32)], [(33, 64)], [(65, 31)],
                                   [(64, 96), (1, 1), (33, 5)], [(4, 40), (40, 4), (32, 33), (97, 61)]])
def test_ssim_over_tile_edges_and_ragged_views(sizes):
    g = synth.rng(sum(h * w for h, w in sizes))
    tgts = [g.random((3, h, w)).astype(np.float32) for h, w in sizes]
    imgs = [np.clip(t + g.normal(0, 0.1, t.shape), 0, 1).astype(np.float32) for t in tgts]
    r = _ssim_loss(imgs, tgts)
    total = 0.0
    for v, (x, y) in enumerate(zip(imgs, tgts)):
        s, grad = oracle.ssim(x, y)
        total += 1.0 - s
        got = r.g_rgb[:, r.pix_off[v]:r.pix_off[v + 1]].cpu().numpy().reshape(x.shape)
        # a sum of 121 window terms over f32 moments: 1e-4 of the largest
        np.testing.assert_allclose(got, -grad, atol=1e-4 * np.abs(grad).max())
    # per view a mean of quotients of differences of f32 moments (at most 1, two times eleven taps) over denominators of
    # 9e-4 and up
    assert r.loss_out[0].item() == pytest.approx(total, abs=len(sizes) * 64 * 2.0 ** -24 / 9e-4)


@pytest.mark.parametrize("shift", [1, 2, 3, 29])
def test_ssim_sum_does_not_depend_on_the_grouping_of_its_values(shift):
    """Content on black moved by `shift` rows has the same values of S, in other groups of a thread's four rows: summed
    in f64 (each value is an f32) the totals differ by f64 rounding alone."""
    g = synth.rng(3)
    H, W = 160, 96
    totals = []
    y = g.random((3, 64, W)).astype(np.float32)
    x = np.clip(y + g.normal(0, 0.05, y.shape), 0, 1).astype(np.float32)
    for top in (32, 32 + shift):
        canvas = np.zeros((2, 3, H, W), np.float32)
        canvas[0, :, top:top + 64], canvas[1, :, top:top + 64] = x, y
        totals.append(_ssim_loss([canvas[0]], [canvas[1]]).loss_out[0].item())
    # 3 H W additions of values of at most 1, each rounded at 2^-53 of a sum of at most 3 H W, in a mean of 3 H W
    assert abs(totals[0] - totals[1]) <= 2 * 3 * H * W * 2.0 ** -53
