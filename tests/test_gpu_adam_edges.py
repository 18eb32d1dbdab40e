"""The mapping update's root and quotient where their correction step does not apply (zero, denormal,
huge, infinite and NaN moments, eps 0) and around the edges of its range, against IEEE f32 operations (GPU)."""
import numpy as np
import pytest
import torch

from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu

VALUES = np.array([0.0, 1e-45, 1e-40, 1.2e-38, 9e-37, 1.1e-36, 1e-30, 1e-20, 3e-9, 1e-4, 0.7, 33.0, 1e10, 9e35, 1.1e36,
                   1e38, np.inf, np.nan], np.float32)


@pytest.mark.parametrize("eps", [1e-15, 1e-8, 0.0])
@pytest.mark.parametrize("device_count", [False, True])
def test_update_of_special_moments(eps, device_count):
    m0, v0 = (a.ravel() for a in np.meshgrid(np.concatenate([VALUES, -VALUES]), VALUES))
    n = m0.size
    f = raster.Field(*(torch.zeros(n, k, device="cuda") for k in (3, 4, 3)), torch.zeros(n, device="cuda"),
                     torch.zeros(n, 3, device="cuda"), torch.zeros(n, 0, device="cuda"))
    opt = raster.MappingAdam(f, eps=eps)
    for half, x in ((0, m0), (1, v0)):  # the opacity group: after means (3 n), quats (4 n), log-scales (3 n)
        opt.moments[half * 14 * n + 10 * n:][:n].copy_(torch.as_tensor(x))
    r = raster.Renderer(n, [synth.camera(16, 16, 16.0)], 0, 64)
    t = 7
    opt.step_ctr.fill_(float(t - 1))
    opt.step(r, 0 if device_count else t)
    got = f.opacity_logits.cpu().numpy()
    with np.errstate(all="ignore"):
        m, v = np.float32(0.9) * m0, np.float32(0.999) * v0
        mh, vh = m / np.float32(1 - 0.9 ** t), v / np.float32(1 - 0.999 ** t)
        want = -(np.float32(opt.lr[3]) * mh / (np.sqrt(vh) + np.float32(eps)))
    # an overflow of an intermediate result may be reached a rounding earlier or later
    clear = ~(np.isfinite(m0) & (np.abs(m0) > 1e37)) & ~(np.isfinite(v0) & (v0 > 1e37))
    got, want = got[clear], want[clear].astype(np.float32)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    ok = np.isfinite(want)
    # four f32 roundings on each side (bias corrections, product, root, quotient), and the smallest denormals
    assert (np.abs(got[ok].astype(np.float64) - want[ok]) <= 8 * 2.0 ** -24 * np.abs(want[ok]) + 2e-44).all()
    assert opt.step_ctr.item() == (t if device_count else t - 1)
