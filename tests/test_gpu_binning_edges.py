"""Binning at the edges of its chunk sizes and digit widths, bit-exact against the definition: images whose tile
counts need digits of 5 to 8 bits in one and two passes, item counts around the scan, depth and emission
chunks, splats that cover every tile, centres far outside the image (GPU)."""
import numpy as np
import pytest
import torch

import gpu_cases as C
import oracle
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu


def _check(r, gs, cams):
    torch.cuda.synchronize()
    assert r.status() == 0
    keys, vals, ranges = C.gpu_binning(r)
    uvdo, conic, touched = (t.cpu().numpy() for t in (r.uvdo, r.conic, r.touched))
    want_k, want_v, tile0 = [], [], 0
    for v, cam in enumerate(cams):
        sl = slice(v * gs.n, (v + 1) * gs.n)
        rect, _ = oracle.rects(uvdo[sl, :2].astype(np.float64), conic[sl, 3].astype(np.int32), cam.width, cam.height, 16)
        TX, TY = -(-cam.width // 16), -(-cam.height // 16)
        area = (rect[:, 2] - rect[:, 0]) * (rect[:, 3] - rect[:, 1])
        vis = conic[sl, 3] > 0
        assert np.array_equal(touched[sl], np.where(vis, area, 0))
        who = np.repeat(np.arange(gs.n)[vis], area[vis])
        j = np.arange(who.size) - np.repeat(np.cumsum(area[vis]) - area[vis], area[vis])
        w = np.maximum(rect[who, 2] - rect[who, 0], 1)
        want_k.append((tile0 + (rect[who, 1] + j // w) * TX + rect[who, 0] + j % w).astype(np.uint64) << np.uint64(32)
                      | uvdo[sl][who, 2].view(np.uint32))
        want_v.append((who + v * gs.n).astype(np.uint32))
        tile0 += TX * TY
    k, i = np.concatenate(want_k), np.concatenate(want_v)
    order = np.lexsort((i, k))
    assert np.array_equal(keys, k[order]) and np.array_equal(vals, i[order])
    tile = (k[order] >> np.uint64(32)).astype(np.int64)
    count = np.bincount(tile, minlength=tile0)
    end = np.cumsum(count)
    assert np.array_equal(ranges[:, 1], np.where(count > 0, end, 0)) and np.array_equal(ranges[:, 0], np.where(count > 0, end - count, 0))
    order = r.tile_order.cpu().numpy()
    assert np.array_equal(np.sort(order), np.arange(tile0))


# tiles: 1, 16, 17 (5 bits), 64, 65 (7), 256, 272 (two passes of 5), 1024 and 1056 (5 and 6), 4096, 4160 (7), 16640 (8)
@pytest.mark.parametrize("w,h", [(16, 16), (64, 64), (272, 16), (128, 128), (1040, 16), (256, 256), (272, 256), (512, 512),
                                 (528, 512), (1024, 1024), (1040, 1024), (2080, 2048)])
def test_tile_digit_widths(w, h):
    gs, cam = C.box_case(1500, 4, w, h, 0.9 * w)
    _, r = C.gpu_forward(gs, cam, raster.RasterParams())
    _check(r, gs, [cam])


@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 1024, 1025, 2047, 2048, 2049, 4097])
def test_item_counts_and_views(n):
    gs, cam = C.box_case(n, 4, 200, 120, 150.0)
    cams = [cam, synth.camera(65, 40, 60.0, cx=30, cy=20), synth.camera(64, 48, 60.0, T_cw=np.diag([-1.0, 1.0, -1.0, 1.0]))]
    _, r = C.gpu_forward(gs, cams, raster.RasterParams())
    _check(r, gs, cams)


def test_splats_over_every_tile_and_far_centres():
    """Scales of metres (one item owns whole rounds of the emission), centres up to 1e30 px and a NaN mean."""
    gs, cam = C.box_case(600, 4, 640, 480, 500.0)
    gs.log_scales[:40] = np.float32(0.5)
    gs.means[40:60, 0] = np.float32([1e3, -1e3, 1e6, -1e6, 1e9, -1e9, 1e20, -1e20, 1e28, -1e28] * 2)
    gs.means[60] = np.nan
    _, r = C.gpu_forward(gs, cam, raster.RasterParams())
    _check(r, gs, [cam])


def test_more_than_one_wave_of_chunks():
    """Depth and tile passes with several times as many chunks as resident blocks."""
    room = synth.make_room(0)
    gs = synth.room_field(400_000, 4, room=room)
    cams = [synth.room_camera(1200, 680, 600.0, room=room)] * 6
    _, r = C.gpu_forward(gs, cams, raster.RasterParams())
    assert r.instances() > 4096 * 152 * 3 * 2
    _check(r, gs, cams)


# more than 2^21 (view, Gaussian) items: chunks of 2,048 items and their look-back flags cleared by the compaction, few and
# many of them visible, on buffers that an earlier call has filled
@pytest.mark.parametrize("facing", [True, False])
def test_many_items_of_which_few_are_visible(facing):
    gs, cam = C.box_case(270_000, 4, 64, 48, 60.0)
    away = synth.camera(64, 48, 60.0, T_cw=np.diag([-1.0, 1.0, -1.0, 1.0]))
    cams = [cam] * 8 if facing else [away, cam] + [away] * 6
    gs.log_scales[:] -= 3.0   # small splats: the instances stay few
    field, r = C.gpu_forward(gs, cams, raster.RasterParams())
    _check(r, gs, cams)
    r.project(field)
    r.bin_sort(want_keys=True)
    _check(r, gs, cams)
