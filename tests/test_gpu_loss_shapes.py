"""The loss kernel at the edges of its class bounds (8, 16, 24, 32), with every feature width, in mapping and
tracking mode, over views of different sizes (whole blocks, less than a warp, ragged), against the oracle;
the tracking median over views without any depth (GPU)."""
import numpy as np
import pytest
import torch

import gpu_cases as C
import oracle
from paper_2603_27781_gb300 import raster, synth

pytestmark = pytest.mark.gpu

SIZES = ((48, 64), (5, 7), (33, 97))


@pytest.mark.parametrize("mode", ["mapping", "tracking"])
@pytest.mark.parametrize("D,K", [(4, 1), (4, 24), (8, 9), (8, 24), (16, 8), (16, 16), (16, 17), (16, 24), (16, 25), (32, 7),
                                 (32, 8), (32, 16), (32, 24), (32, 32)])
def test_loss_over_ragged_views(D, K, mode):
    g = synth.rng(100 * D + K)
    cams = [synth.camera(w, h, 60.0) for h, w in SIZES]
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    imgs = [dict(rgb=f32(g.random((3, h, w))), depth=f32(g.uniform(2, 5, (h, w))), sil=f32(g.uniform(0.97, 1.0, (h, w))),
                 feat=f32(g.standard_normal((D, h, w)))) for h, w in SIZES]
    tgts = [synth.Frame(g.random((3, h, w)).astype(np.float32),
                        (im["depth"] + g.normal(0, 0.05, (h, w)) * (g.random((h, w)) < 0.9)).astype(np.float32),
                        g.integers(0, K, (h, w)).astype(np.uint8)) for im, (h, w) in zip(imgs, SIZES)]
    for t in tgts:
        t.depth[0, :3] = 0.0
        t.label[1, :4] = 255
    dec = synth.decoder(K, D, seed=K)
    w = raster.MAPPING if mode == "mapping" else raster.TRACKING
    wo = oracle.MAPPING if mode == "mapping" else oracle.TRACKING
    r = raster.Renderer(0, cams, D, 0, n_classes=K)
    flat = lambda xs: torch.as_tensor(np.concatenate(xs, -1)).cuda()
    for k in ("rgb", "depth", "sil", "feat"):
        t = getattr(r, "img_" + k)
        t.copy_(flat([im[k].reshape(*t.shape[:-1], -1) for im in imgs]))
    tg = dict(rgb=flat([t.rgb.reshape(3, -1) for t in tgts]), depth=flat([t.depth.ravel() for t in tgts]),
              label=flat([t.label.ravel() for t in tgts]))
    r.loss(tg, torch.as_tensor(dec.W).cuda(), torch.as_tensor(dec.b).cuda(), w)
    total, dW, db = 0.0, 0.0, 0.0
    for v, (im, t) in enumerate(zip(imgs, tgts)):
        o = oracle.loss(im, t, dec, wo)
        a, b = r.pix_off[v], r.pix_off[v + 1]
        if mode == "tracking":
            e = np.abs(im["depth"].astype(np.float32) - t.depth)[t.depth > 0]
            assert r.median[v].item() == np.float32(oracle.lower_median(e.astype(np.float64)))
        for k, tol in (("rgb", 1e-9), ("depth", 1e-9), ("feat", 1e-9)):
            got = getattr(r, "g_" + k)[..., a:b].cpu().numpy().reshape(o[k].shape)
            np.testing.assert_allclose(got, o[k], atol=tol, rtol=1e-5)
        total, dW, db = total + o["total"], dW + o["W"], db + o["b"]
    assert r.loss_out[0].item() == pytest.approx(total, rel=1e-5)
    C.assert_grad_close("dW", r.d_dec_W.cpu().numpy(), dW, 1e-5)
    C.assert_grad_close("db", r.d_dec_b.cpu().numpy(), db, 1e-5)


@pytest.mark.parametrize("D,K", [(0, 0), (16, 8), (32, 20)])
def test_views_without_depth_have_no_mask_and_no_gradient(D, K):
    cams = [synth.camera(40, 30, 60.0), synth.camera(33, 17, 60.0)]
    r = raster.Renderer(0, cams, D, 0, n_classes=max(K, 1))
    g = torch.Generator(device="cuda").manual_seed(3)
    r.img_depth.uniform_(1.0, 2.0, generator=g)
    r.img_sil.fill_(1.0)
    r.img_feat.normal_(generator=g)
    depth = torch.zeros(r.P, device="cuda")
    depth[1200:] = r.img_depth[1200:] + 0.01  # the second view has depth everywhere
    tg = dict(rgb=torch.rand(3, r.P, device="cuda", generator=g), depth=depth,
              label=torch.zeros(r.P, dtype=torch.uint8, device="cuda"))
    W, b = (torch.ones(K, D, device="cuda"), torch.zeros(K, device="cuda")) if K else (None, None)
    r.loss(tg, W, b, raster.TRACKING)
    e = (r.img_depth[1200:] - depth[1200:]).abs().sort()[0]
    assert r.median.tolist() == [0.0, e[(len(e) - 1) // 2].item()]
    assert not r.mask[:1200].any() and r.mask[1200:].all()
    assert not r.g_rgb[:, :1200].any() and not r.g_depth[:1200].any() and not r.g_feat[:, :1200].any()
    assert r.g_rgb[:, 1200:].all() and r.g_depth[1200:].all()
