"""The one-view projection, which lists a block's Gaussians in front of the camera, equals the projection of several
views, which does not, bit for bit: at the edges of its 256-Gaussian blocks, with all, some and none in front, with
zero quaternions and non-finite means (GPU)."""
import numpy as np
import pytest
import torch

import gpu_cases as C
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 512, 1000])
@pytest.mark.parametrize("where", ["front", "mixed", "behind"])
def test_one_view_equals_several(n, where):
    gs, cam = C.box_case(n, 4, 64, 48, 60.0)
    if where != "front":
        cam = synth.camera(64, 48, 60.0, T_cw=np.diag([-1.0, 1.0, -1.0, 1.0]))
    if where == "mixed":
        gs.means[::2, 2] *= -1.0
        gs.means[n // 2, 0] = np.nan
        gs.means[n // 3, 2] = np.inf
        gs.quats[n // 4] = 0.0
    field = raster.Field.from_numpy(gs)
    one, two = (raster.Renderer(n, [cam] * k, 4, 64) for k in (1, 2))
    for pose in (None, torch.tensor(np.asarray(cam.T_cw), dtype=torch.float32, device="cuda").reshape(1, 16)):
        one.project(field, pose)
        two.project(field, None if pose is None else pose.repeat(2, 1).contiguous())
        torch.cuda.synchronize()
        for k in ("uvdo", "uv_lo", "conic", "touched"):
            a, b = getattr(one, k).view(torch.int32), getattr(two, k).view(torch.int32)
            assert torch.equal(a, b[:n]) and torch.equal(a, b[n:]), k
        assert where == "front" or int((one.touched > 0).sum()) < n
