"""The joint copies around the autograd function and the expansion: every form of image gradient that
autograd can hand over reaches the renderer's buffers, and a field under autograd grows as one without (GPU)."""
import numpy as np
import pytest
import torch

import gpu_cases as C
from paper_2603_27781_gb300 import raster

pytestmark = pytest.mark.gpu

ARRAYS = ("means", "quats", "log_scales", "opacity_logits", "rgb", "feat")


@pytest.mark.parametrize("d", [0, 8])
@pytest.mark.parametrize("form", ["dense", "absent", "expanded", "strided", "create_graph"])
def test_image_gradients_of_every_form(d, form):
    gs, cam = C.box_case(500, d, 67, 45, 60.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    leaves = [getattr(field, k).clone().requires_grad_(True) for k in ARRAYS]
    outs = raster.rasterize(r, *leaves)
    for o, buf in zip(outs, (r.img_rgb, r.img_depth, r.img_sil, r.img_feat[:d])):
        assert torch.equal(o, buf) and o.data_ptr() != buf.data_ptr() or o.numel() == 0
    g = torch.Generator(device="cuda").manual_seed(2)
    grads = [torch.randn(o.shape, generator=g, device="cuda") for o in outs]
    if form == "expanded":
        grads = [torch.full((1,) * o.dim(), 0.25 + i, device="cuda").expand(o.shape) for i, o in enumerate(outs)]
    elif form == "strided":
        grads = [torch.randn(tuple(reversed(o.shape)), generator=g, device="cuda").T if o.dim() == 2 else
                 torch.randn(2 * o.numel(), generator=g, device="cuda")[1::2] for o in outs]
    use = [0, 2] if form == "absent" else [i for i in range(4) if outs[i].numel()]
    got = torch.autograd.grad([outs[i] for i in use], leaves[:5], [grads[i] for i in use],
                              create_graph=form == "create_graph")
    for i, buf in enumerate((r.g_rgb, r.g_depth, r.g_sil, r.g_feat[:d])):
        assert torch.equal(buf, grads[i] if i in use else torch.zeros_like(buf)) and not buf.requires_grad
    for x, buf in zip(got, (r.d_means, r.d_quats, r.d_log_scales, r.d_logits, r.d_rgb)):
        assert torch.equal(x, buf) and x.data_ptr() != buf.data_ptr()


def test_expansion_of_a_field_under_autograd():
    gs, cam = C.box_case(300, 4, 48, 32, 40.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    P = r.P
    tg = dict(rgb=torch.rand(3, P, device="cuda"), depth=torch.full((P,), 1.5, device="cuda"),
              label=torch.zeros(P, dtype=torch.uint8, device="cuda"))
    feat = torch.randn(P, 4, device="cuda")
    plain, src, total, status = raster.expand(r, field, tg, feat)
    leaves = raster.Field(*(getattr(field, k).clone().requires_grad_(True) for k in ARRAYS))
    grown, src2, total2, status2 = raster.expand(r, leaves, tg, feat)
    assert (total, status) == (total2, status2) and status == 0 and total > 0 and torch.equal(src, src2)
    for k in ARRAYS:
        a, b = getattr(plain, k), getattr(grown, k)
        assert torch.equal(a, b.detach()) and a.shape[0] == gs.n + total and not a.requires_grad
        w = torch.randn_like(a)
        (x,) = torch.autograd.grad(b, getattr(leaves, k), w)
        np.testing.assert_array_equal(x.cpu().numpy(), w[: gs.n].cpu().numpy())
