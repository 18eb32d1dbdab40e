"""Expansion on a stream of the caller's own: the count is read when that stream has written it (GPU)."""
import pytest
import torch

import gpu_cases as C
from paper_2603_27781_gb300 import raster

pytestmark = pytest.mark.gpu


def test_expansion_on_a_busy_side_stream():
    gs, cam = C.box_case(300, 4, 48, 32, 40.0)
    field, r = C.gpu_forward(gs, cam, raster.RasterParams())
    tg = dict(rgb=torch.rand(3, r.P, device="cuda"), depth=torch.full((r.P,), 1.5, device="cuda"),
              label=torch.zeros(r.P, dtype=torch.uint8, device="cuda"))
    feat = torch.randn(r.P, 4, device="cuda")
    want, src, total, status = raster.expand(r, field, tg, feat)
    assert total > 0 and status == 0
    side = torch.cuda.Stream()
    for delay in (0, 20_000_000):       # cycles that the side stream is busy for before the call's work
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(delay)
        out, src2, total2, status2 = raster.expand(r, field, tg, feat, stream=side)
        assert (total2, status2) == (total, status) and torch.equal(src2, src)
        for k in ("means", "quats", "log_scales", "opacity_logits", "rgb", "feat"):
            assert torch.equal(getattr(out, k), getattr(want, k))
