"""The launch shapes that the library picks by itself: on both sides of each line where the default
number of pixels per thread changes with the tile count, the images equal those of the explicit shapes
bit for bit and the gradients agree to the rounding of their sums (GPU)."""
import dataclasses

import pytest
import torch

import gpu_cases as C
from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster

pytestmark = pytest.mark.gpu

IMAGES = ("img_rgb", "img_depth", "img_sil", "img_feat", "img_T", "img_nc", "blend_mask")
# float atomics in another order and sums split over other lanes: a few 1e-6 of the norm; the geometric sums
# pass through the splats' conics, so they are held to the gradient tolerance of the parity tests
SUMS = {"sg_rgb": 1e-5, "d_feat": 1e-5, "sg_uvod": C.TOL_GRAD, "sg_conic": C.TOL_GRAD}


def _shape(r, **kw):
    r.prm_c = dataclasses.replace(r.params, **kw).c()


# forward: 1824 tiles at D = 16, 1216 at D = 32; backward at D = 16 and 32: 912, 608 (map, factored), 1216, 912 (map,
# features), 1216, 760 (pose)
@pytest.mark.parametrize("d,w,h", [(16, 16, 16), (16, 17, 33), (16, 304, 224), (16, 299, 219), (16, 608, 384),
                                   (16, 600, 391), (16, 640, 480), (16, 641, 497), (32, 33, 16), (32, 304, 224),
                                   (32, 640, 304), (32, 641, 305), (32, 608, 512), (32, 600, 521),
                                   (16, 912, 512), (16, 900, 529), (16, 601, 390), (32, 608, 256), (32, 601, 255),
                                   (32, 608, 384), (32, 595, 377)])
def test_default_shapes_match_the_explicit_ones(d, w, h):
    gs, cam = C.box_case(3000, d, w, h, 0.9 * w)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams(), n_classes=8)
    ref = {k: getattr(r, k).clone() for k in IMAGES}
    g = torch.Generator(device="cuda").manual_seed(1)
    for t in (r.g_rgb, r.g_depth, r.g_sil, r.g_feat, r.g_coef):
        t.copy_(torch.randn(t.shape, generator=g, device="cuda"))
    r._basis = torch.randn(8, d, generator=g, device="cuda")
    for np_ in (1, 2):
        for kw in (dict(fwd_px_per_thread=np_), dict(fwd_px_per_thread=np_, fwd_blocks=L.GS_BWD_BLOCKS_GROUP)):
            _shape(r, **kw)
            r.render_fwd(field)
            for k in IMAGES:
                assert torch.equal(getattr(r, k), ref[k]), (kw, k)
    for factored in (False, True):
        for mode in (L.GS_GRAD_MAP, L.GS_GRAD_POSE):
            names = SUMS if mode == L.GS_GRAD_MAP else ("sg_uvod", "sg_conic")
            _shape(r)
            r.render_bwd(field, mode, factored=factored)
            want = {k: getattr(r, k).double() for k in names}
            for np_ in (1, 2):
                _shape(r, bwd_px_per_thread=np_, bwd_blocks=L.GS_BWD_BLOCKS_GROUP)
                r.render_bwd(field, mode, factored=factored)
                for k in names:
                    err = (getattr(r, k).double() - want[k]).norm() / want[k].norm()
                    assert err <= SUMS[k], (factored, mode, np_, k, float(err))
    assert r.status() == 0


def test_default_pixels_with_another_batch_stay_accepted():
    """A staged batch of 64 or 256 is built for two pixels per thread only: asking for one with the
    default pixels per thread on a small image still takes that shape."""
    gs, cam = C.box_case(2000, 16, 64, 48, 60.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    ref = r.img_feat.clone()
    for batch in (64, 256):
        _shape(r, fwd_batch=batch)
        r.render_fwd(field)
        assert torch.equal(r.img_feat, ref)
    _shape(r, fwd_blocks=L.GS_BLOCKS_RING, fwd_batch=64)
    r.render_fwd(field)
    assert torch.equal(r.img_feat, ref)
    assert r.status() == 0
