"""Forward-mode differentiation around the library's calls: tensors with tangents are taken where plain ones are (GPU)."""
import pytest
import torch
import torch.autograd.forward_ad as fwd

import gpu_cases as C
from paper_2603_27781_gb300 import raster

pytestmark = pytest.mark.gpu

ARRAYS = ("means", "quats", "log_scales", "opacity_logits", "rgb", "feat")


def test_expansion_of_a_field_with_tangents():
    """The old Gaussians keep their tangents, the new ones have none."""
    gs, cam = C.box_case(300, 4, 48, 32, 40.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    tg = dict(rgb=torch.rand(3, r.P, device="cuda"), depth=torch.full((r.P,), 1.5, device="cuda"),
              label=torch.zeros(r.P, dtype=torch.uint8, device="cuda"))
    feat = torch.randn(r.P, 4, device="cuda")
    plain, _, total, _ = raster.expand(r, field, tg, feat)
    assert total > 0
    with fwd.dual_level():
        tangents = [torch.randn_like(getattr(field, k)) for k in ARRAYS]
        dual = raster.Field(*(fwd.make_dual(getattr(field, k), t) for k, t in zip(ARRAYS, tangents)))
        grown, _, total2, status = raster.expand(r, dual, tg, feat)
        assert (total2, status) == (total, 0)
        for k, t in zip(ARRAYS, tangents):
            x, xt = fwd.unpack_dual(getattr(grown, k))
            assert torch.equal(x, getattr(plain, k))
            assert torch.equal(xt[: gs.n], t) and not xt[gs.n:].any()


def test_backward_from_image_gradients_with_tangents():
    """The rasterizer's backward has no second derivative: it takes such gradients by their values."""
    gs, cam = C.box_case(500, 8, 67, 45, 60.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    leaves = [getattr(field, k).clone().requires_grad_(True) for k in ARRAYS]
    outs = raster.rasterize(r, *leaves)
    grads = [torch.randn_like(o) for o in outs]
    want = torch.autograd.grad(outs, leaves, grads, retain_graph=True)
    with fwd.dual_level():
        duals = [fwd.make_dual(g, torch.ones_like(g)) for g in grads]
        got = torch.autograd.grad(outs, leaves, duals)
        for a, b in zip(got, want):
            a = fwd.unpack_dual(a).primal
            # float atomics in any order
            assert torch.allclose(a, b, rtol=1e-4, atol=1e-5 * float(b.abs().max()))
    for buf, g in zip((r.g_rgb, r.g_depth, r.g_sil, r.g_feat), grads):
        assert torch.equal(buf, g)
