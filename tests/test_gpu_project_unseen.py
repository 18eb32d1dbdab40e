"""Gradients of Gaussians that no view sees and whose parameters overflow or are not numbers: zero, with one view and with
several (GPU)."""
import numpy as np
import pytest
import torch

import gpu_cases as C
from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views", [1, 3])
@pytest.mark.parametrize("D", [0, 16])
def test_broken_unseen_gaussians_have_no_gradient(views, D):
    gs, cam = C.box_case(400, D, 64, 48, 60.0)
    gs.log_scales[:10] = 90.0           # exp overflows: no finite covariance
    gs.log_scales[10:20] = np.nan
    gs.quats[20:30] = np.nan
    gs.quats[30:40] = 0.0
    gs.means[40:50] = np.inf
    field, r = C.gpu_forward(gs, [cam] * views, raster.RasterParams())
    assert not r.touched.view(views, gs.n)[:, :50].any()
    for buf in (r.g_rgb, r.g_depth, r.g_sil, r.g_feat):
        buf.normal_(generator=torch.Generator(device="cuda").manual_seed(1))
    r.backward(field, L.GS_GRAD_MAP | L.GS_GRAD_POSE)
    for x in (r.d_means, r.d_quats, r.d_log_scales, r.d_logits, r.d_rgb, r.d_feat):
        assert not x[:50].any() and x.isfinite().all()
    assert r.d_twist.isfinite().all() and r.d_means[50:].any()
