"""The mapping update's root and quotient are the IEEE ones, bit for bit, over the whole range of moments (GPU)."""
import numpy as np
import pytest
import torch

from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu


def _moments(kind, n, g):
    mant = 1.0 + g.random(n)
    sign = np.where(g.random(n) < 0.5, -1.0, 1.0)
    if kind == "training":      # what a mapping run holds, and moments that decay out of view
        m, v = 10.0 ** g.uniform(-12, 0, n), 10.0 ** g.uniform(-20, 0, n)
    elif kind == "decayed":
        m, v = 10.0 ** g.uniform(-45, -20, n), 10.0 ** g.uniform(-45, -25, n)
    else:                       # any exponent, denormals included
        m, v = mant * 2.0 ** g.integers(-149, 120, n), mant * 2.0 ** g.integers(-149, 120, n)
    zero = g.random((2, n)) < 0.02
    return (np.where(zero[0], 0.0, sign * m).astype(np.float32), np.where(zero[1], 0.0, v).astype(np.float32))


@pytest.mark.parametrize("eps", [1e-15, 1e-8, 0.0])
@pytest.mark.parametrize("kind", ["training", "decayed", "any"])
def test_update_equals_ieee_operations(kind, eps):
    n, t = 1 << 18, 7
    m0, v0 = _moments(kind, n, synth.rng(5))
    f = raster.Field(*(torch.zeros(n, k, device="cuda") for k in (3, 4, 3)), torch.zeros(n, device="cuda"),
                     torch.zeros(n, 3, device="cuda"), torch.zeros(n, 0, device="cuda"))
    opt = raster.MappingAdam(f, eps=eps)
    for half, x in ((0, m0), (1, v0)):  # the opacity group: after means (3 n), quats (4 n), log-scales (3 n)
        opt.moments[half * 14 * n + 10 * n:][:n].copy_(torch.as_tensor(x))
    opt.step(raster.Renderer(n, [synth.camera(16, 16, 16.0)], 0, 64), t)
    got = f.opacity_logits.cpu().numpy()
    one = np.float32
    with np.errstate(all="ignore"):
        # zero gradients: the moments' updates are single products; the reciprocal bias corrections rounded once
        m, v = one(0.9) * m0, one(0.999) * v0
        mh, vh = m * one(1.0 / (1.0 - 0.9 ** t)), v * one(1.0 / (1.0 - 0.999 ** t))
        want = one(0) - one(opt.lr[3]) * mh / (np.sqrt(vh) + one(eps))
    assert got.dtype == want.dtype == np.float32
    np.testing.assert_array_equal(got, want)    # NaN (0 / 0 with eps 0) equal to NaN
