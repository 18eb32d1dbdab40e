"""Binning of a caller's own projected records: centres and radii far beyond those that the projection writes, whose tile
rectangles are the definition's (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_27781_gb300 import raster, synth
from test_gpu_binning_edges import _check

pytestmark = pytest.mark.gpu


def test_rectangles_of_far_centres_and_large_radii():
    """Exact in f32 and in 32-bit sums only with care: edges that fall inside the image (a centre 1e8 px away with a
    radius of 1e8 - 320), radii near 2^31, and each of them along x, along y and along both."""
    cam = synth.camera(640, 480, 500.0)
    far = [(100.0, 2.1e9), (300.0, 3e7), (1e8, 1e8 - 320), (-1e8, 1e8 + 304), (7e7, 7e7 - 64), (-7e7, 7e7 + 16), (3e8, 3e8 - 320),
           (-5e8, 5e8 + 352), (1e9, 1e9 - 256), (-1e9, 1e9 + 192), (2e7, 2e7 - 100), (-1.6e7, 1.6e7 + 200)]
    near = 200.0
    rec = [(a, near, r) for a, r in far] + [(near, a, r) for a, r in far] + [(a, a, r) for a, r in far]
    n = len(rec)
    u, v, rad = (np.array(x, np.float32) for x in zip(*rec))
    rect, touched = oracle.rects(np.stack([u, v], 1).astype(np.float64), rad.astype(np.int64).astype(np.int32), 640, 480, 16)
    assert (touched > 0).all() and (touched < 1200).any()
    r = raster.Renderer(n, [cam], 4, int(touched.sum()))
    depth = np.linspace(1.0, 3.0, n, dtype=np.float32)[::-1]
    r.uvdo.copy_(torch.as_tensor(np.stack([u, v, depth, np.full(n, 0.5, np.float32)], 1)))
    r.conic[:, 3] = torch.as_tensor(rad).cuda()
    r.touched.copy_(torch.as_tensor(touched))
    r.bin_sort(want_keys=True)

    class Count:
        pass
    Count.n = n
    _check(r, Count, [cam])
