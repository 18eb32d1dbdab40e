"""The blend backward on the tips of long thin splats, whose alpha there is barely alpha_min: every pixel that the
forward blended takes part, whatever the block form (GPU)."""
import numpy as np
import pytest
import torch

from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu

TILE, GROUP = L.GS_BWD_BLOCKS_TILE, L.GS_BWD_BLOCKS_GROUP
SIZE, F, Z = 96, 600.0, 2.0


def _thin_field(m, D, sigma, seed):
    """m splats of sigma x about 0.55-0.8 px at an angle, most of them with a tip (alpha = alpha_min) in the image; splat i
    has a one in feature channel i (colour channel i without features) and zeros elsewhere."""
    g = synth.rng(seed)
    th = g.uniform(0.1, 1.47, m) + 0.5 * np.pi * g.integers(0, 2, m)
    o = g.uniform(0.02, 0.33, m)
    along = np.sqrt(2.0 * np.log(255.0 * o) * (sigma ** 2 + 0.3))
    uv = g.uniform(0.2 * SIZE, 0.8 * SIZE, (m, 2)) - along[:, None] * np.stack([np.cos(th), np.sin(th)], 1)
    means = np.column_stack([(uv - 0.5 * SIZE) * Z / F, np.full(m, Z) + 0.01 * np.arange(m)])
    means[:, :2] *= means[:, 2:] / Z
    scales = np.column_stack([np.full(m, sigma), g.uniform(0.05, 0.6, m), np.full(m, 1e-3)]) * means[:, 2:] / F
    eye = np.eye(m, dtype=np.float32)
    f32 = lambda a: np.ascontiguousarray(a, np.float32)
    return synth.Gaussians(f32(means), f32(np.column_stack([np.cos(th / 2), 0 * th, 0 * th, np.sin(th / 2)])),
                           f32(np.log(scales)), f32(np.log(o / (1.0 - o))), eye if D == 0 else np.zeros((m, 3), np.float32),
                           eye if D else np.zeros((m, 0), np.float32))


@pytest.mark.parametrize("D,blocks,px,mask", [
    (0, 0, 0, True), (4, 0, 0, True), (8, 0, 0, True), (8, 0, 0, False), (16, TILE, 1, False), (16, TILE, 2, False),
    (16, TILE, 4, False), (16, TILE, 2, True), (32, TILE, 1, False), (32, TILE, 2, False), (16, GROUP, 1, True),
    (16, GROUP, 2, True), (32, GROUP, 2, True)])
@pytest.mark.parametrize("sigma", [300.0, 1000.0])
def test_gradient_reaches_every_blended_pixel_of_a_tip(D, blocks, px, mask, sigma):
    """A channel of the image is the sum of the weights of its one splat, and the gradient of that splat's channel
    under an image gradient of one on a set of pixels is the sum of its weights there: the set holds the pixels of
    weight below 1.05 alpha_min, which no splat may lose."""
    m = D or 3
    cam = synth.camera(SIZE, SIZE, F)
    for seed in range(8):
        gs = _thin_field(m, D, sigma, 1000 * D + seed)
        field = raster.Field.from_numpy(gs)
        r = raster.Renderer(m, [cam], D, m * 36, params=raster.RasterParams(bwd_blocks=blocks, bwd_px_per_thread=px))
        r.use_blend_mask = mask
        r.forward(field)
        image, grad = (r.img_feat, r.g_feat) if D else (r.img_rgb, r.g_rgb)
        weak = (image > 0) & (image < 1.05 / 255.0)
        grad.copy_(weak.float())
        r.backward(field, L.GS_GRAD_MAP)
        assert r.status() == 0
        count = weak.sum(1).cpu().numpy()
        assert count.sum() > 0
        want = (image.double() * weak).sum(1).cpu().numpy()
        got = torch.diagonal(r.d_feat if D else r.d_rgb).cpu().numpy()
        # a weight: up to m recovered transmittances of two divisions' rounding each and the forward's m products; their
        # sum in f32, in any order.  One lost pixel is 1 / (1.05 count) or more of the sum.
        tol = (8 * m + count) * 2.0 ** -24
        assert (1.05 * count * tol < 0.5).all()
        assert (np.abs(got - want) <= tol * want).all(), (seed, count, (got - want) / np.maximum(want, 1e-30))
