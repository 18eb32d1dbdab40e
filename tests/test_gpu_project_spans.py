"""The projection's views per thread and the one-view backward's spans: Gaussian counts around the edges of
both, against the general forms (one view per call; the kernel that loops over views) (GPU)."""
import numpy as np
import pytest
import torch

from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu

GRADS = ("d_means", "d_quats", "d_log_scales", "d_logits", "d_rgb")


def _cams(n):
    return [synth.camera(64, 48, 60.0, cx=32, cy=24, T_cw=synth.perturb_pose(np.eye(4), 3.0 * v, 0.05 * v, seed=v + 1)) for v in range(n)]


# spans of 32, 64 (from 233,472) and 128 (from 466,944) Gaussians per warp, with ragged ends
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000, 233_471, 233_473, 466_943, 467_001])
@pytest.mark.parametrize("mode", [L.GS_GRAD_MAP, L.GS_GRAD_POSE, L.GS_GRAD_MAP | L.GS_GRAD_POSE])
def test_one_view_backward_matches_the_loop_over_views(n, mode):
    field = raster.Field.from_numpy(synth.box_field(n, 0))
    cams = _cams(2)
    one, two = raster.Renderer(n, cams[:1], 0, 0), raster.Renderer(n, cams, 0, 0)
    g = torch.Generator(device="cuda").manual_seed(n)
    seen = torch.rand(n, 1, generator=g, device="cuda") < 0.2
    for k in ("sg_uvod", "sg_conic", "sg_rgb"):
        x = torch.randn(n, 4, generator=g, device="cuda") * seen
        getattr(one, k).copy_(x)
        getattr(two, k).zero_()
        getattr(two, k)[:n].copy_(x)
    one.sg_rgb[-1] = two.sg_rgb[-1] = 1.0  # a colour gradient without a geometric one
    for r in (one, two):
        for k in GRADS + ("pose_part",):
            getattr(r, k).fill_(7.0)
        r.project_bwd(field, mode)
    if mode & L.GS_GRAD_MAP:
        for k in GRADS:
            a, b = getattr(one, k), getattr(two, k)
            # the same operations, contracted differently at most: a few ulp of the largest terms
            assert (a - b).norm() <= 1e-6 * b.norm(), k
            assert torch.equal(a[~seen[:, 0]] == 0, b[~seen[:, 0]] == 0), k
    else:
        assert all((getattr(one, k) == 7.0).all() for k in GRADS)
    if mode & L.GS_GRAD_POSE:
        assert (one.pose_part[0] - two.pose_part[0]).norm() <= 1e-6 * two.pose_part[0].norm()
        assert not two.pose_part[1].any() and not one.pose_part[0][:, ~seen[:, 0]].any()
    else:
        assert (one.pose_part == 7.0).all()


@pytest.mark.parametrize("n,views", [(1, 3), (257, 5), (90_001, 8), (120_000, 7), (330_000, 3)])
def test_projection_of_several_views_is_that_of_each(n, views):
    """Groups of views per thread: all of them, some, one; bit for bit what one view per call gives."""
    field = raster.Field.from_numpy(synth.box_field(n, 0))
    cams = _cams(views)
    r = raster.Renderer(n, cams, 0, 0)
    r.project(field)
    for v, cam in enumerate(cams):
        o = raster.Renderer(n, [cam], 0, 0)
        o.project(field)
        for k in ("uvdo", "uv_lo", "conic", "touched"):
            assert torch.equal(getattr(r, k)[v * n:(v + 1) * n], getattr(o, k)), (v, k)
