"""The work that programs built on this framework have it do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" says which public entry point it goes through:

  step      one forward + backward pass of the whole path (`Renderer.iteration`), replayed from a CUDA
            graph that the program captured once, as the mapping loop and the benchmark run it
  track     one frame tracked against a fixed map (`Tracker.track`)
  render    one forward pass, launched eagerly (`Renderer.forward`), as for evaluation
  autograd  forward and backward through `torch.autograd` (`rasterize`), launched eagerly
  bin       projection, binning and sort of a batch of keyframes (`Renderer.project`, `bin_sort`)
  loss      decoder, losses and image gradients (`Renderer.loss`)
  adam      the mapping update (`MappingAdam.step`)
  expand    the growth of the map by a frame's unobserved pixels (`expand`)

Scenes: "box" (Gaussians in a box before the camera, the small test scene), "room" (Gaussians on the
surfaces of a furnished room, the benchmark's scene) and "scan" (Gaussians unprojected from depth frames of
that room, about as large as their pixels: the map that the SLAM loop builds).  Observations are rays cast
into the room.  `exact` is the method in float64 torch, written from the paper's equations.
"""
import math

import numpy as np
import torch

from paper_2603_27781_gb300 import _lib as L
from paper_2603_27781_gb300 import raster, slam, synth

DEV = "cuda"
GROUPS = ("means", "quats", "log_scales", "opacity_logits", "rgb", "feat")


def listed():
    return [
        # The smallest call: the 2,000-Gaussian test scene, one mapping and pose gradient; latency and launches.
        dict(name="step_tiny", kind="step", scene="box", n=2000, d=16, k=8, w=64, h=48, fx=60.0, views=1, ragged=False,
             half=False, pose=True, ssim=0.0),
        # The benchmark's frame: a room-scale map at Replica's resolution, map and pose gradients.
        dict(name="step_room", kind="step", scene="room", n=1_000_000, d=16, k=8, w=1200, h=680, fx=600.0, views=1,
             ragged=False, half=False, pose=True, ssim=0.0),
        # The wide-feature map at ScanNet's resolution, gradients of the map alone.
        dict(name="step_vga_d32", kind="step", scene="room", n=1_000_000, d=32, k=8, w=640, h=480, fx=525.0, views=1,
             ragged=False, half=False, pose=False, ssim=0.0),
        # One mapping iteration of the SLAM loop: the keyframe draw, then the mapping loss with its SSIM term on the
        # map that a scan has built.
        dict(name="step_slam", kind="step", scene="scan", n=850_000, d=16, k=8, w=1200, h=680, fx=600.0, views=1,
             ragged=False, half=False, pose=False, ssim=0.2),
        # The largest: a batch of eight keyframes of two resolutions against a 2M-Gaussian map in 16-bit storage.
        dict(name="step_batch_half", kind="step", scene="room", n=2_000_000, d=32, k=8, w=1200, h=680, fx=600.0, views=8,
             ragged=True, half=True, pose=True, ssim=0.0),
        # A tracked frame: 40 pose-only iterations from the constant-velocity start.
        dict(name="track", kind="track", scene="scan", n=300_000, d=16, k=8, w=1200, h=680, fx=600.0, iters=40),
        # A rendered view for evaluation: odd size, a feature width that the mapping cases do not use.
        dict(name="render_odd_d8", kind="render", scene="room", n=300_000, d=8, w=811, h=607, fx=421.0),
        # A PyTorch program with a loss of its own: dense image gradients through the autograd function.
        dict(name="autograd_d16", kind="autograd", scene="room", n=100_000, d=16, w=640, h=480, fx=525.0),
        # The geometry of a mapping batch of keyframes: projection, binning and sort.
        dict(name="bin_keyframes", kind="bin", scene="room", n=1_000_000, w=1200, h=680, fx=600.0, views=6, ragged=True),
        # The mapping loss of a frame with 20 classes, with the gradient of the features themselves.
        dict(name="loss_k20", kind="loss", d=16, k=20, w=1200, h=680, views=1, ragged=False, mask=False),
        # The mapping update of the benchmark's map.
        dict(name="adam_room", kind="adam", n=1_000_000, d=16),
        # A new keyframe with about a tenth of its pixels unobserved.
        dict(name="expand_frame", kind="expand", n=300_000, d=16, w=1200, h=680, fx=600.0, unseen=0.1),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    size = lambda lo, hi: dict(w=log(lo, hi), h=log(max(16, lo * 3 // 5), hi * 3 // 5))
    kind = rng.choice(("step", "step", "step", "track", "render", "autograd", "bin", "loss", "adam", "expand"))
    if kind == "adam":
        return dict(kind=kind, n=log(1000, 1_500_000), d=rng.choice((0, 8, 16, 32)))
    if kind == "loss":
        d, k = rng.choice((4, 8, 16, 32)), rng.choice((rng.randint(2, 8), rng.randint(9, 32)))
        return dict(kind=kind, d=d, k=k, views=rng.choice((1, 1, 2, 4)), ragged=rng.random() < 0.5,
                    mask=d <= 16 and k <= 8 and rng.random() < 0.7, **size(64, 1280))
    if kind == "expand":
        s = size(160, 1280)
        return dict(kind=kind, n=log(2000, 800_000), d=rng.choice((0, 8, 16, 32)), fx=rng.uniform(0.5, 0.9) * s["w"],
                    unseen=rng.uniform(0.0, 0.4), **s)
    if kind == "bin":
        s = size(160, 1280)
        return dict(kind=kind, scene=rng.choice(("room", "scan")), n=log(2000, 1_500_000), views=rng.choice((1, 2, 4, 6)),
                    ragged=rng.random() < 0.5, fx=rng.uniform(0.5, 0.9) * s["w"], **s)
    if kind == "track":
        s = size(160, 1280)
        return dict(kind=kind, scene="scan", n=log(10_000, 600_000), d=16, k=rng.randint(2, 8), iters=rng.choice((10, 20, 40)),
                    fx=rng.uniform(0.5, 0.9) * s["w"], **s)
    if kind == "step":
        s = size(64, 1280)
        views = rng.choice((1, 1, 1, 2, 3, 4))
        d = rng.choice((8, 16, 16, 32))
        return dict(kind=kind, scene=rng.choice(("box", "room", "scan")), n=log(2000, 1_500_000), d=d, k=rng.randint(2, 8),
                    views=views, ragged=views > 1 and rng.random() < 0.5, half=d >= 16 and rng.random() < 0.3,
                    pose=rng.random() < 0.5, ssim=rng.choice((0.0, 0.2)), fx=rng.uniform(0.5, 0.9) * s["w"], **s)
    s = size(64, 1280)
    return dict(kind=kind, scene=rng.choice(("box", "room", "scan")), n=log(2000, 1_000_000),
                d=rng.choice((4, 8, 16, 32)), fx=rng.uniform(0.5, 0.9) * s["w"], **s)


# ------------------------------------------------------------------------------------- inputs
def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + salt)


def _rays(room, cam):
    """Depth, colour and class of the room's surfaces along a camera's pixel rays (float64 [P], [3,P], [P])."""
    t64 = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)
    H, W = cam.height, cam.width
    py, px = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64), torch.arange(W, device=DEV, dtype=torch.float64),
                            indexing="ij")
    dc = torch.stack([(px + 0.5 - cam.cx) / cam.fx, (py + 0.5 - cam.cy) / cam.fy, torch.ones_like(px)], -1).reshape(-1, 3)
    T = t64(cam.T_cw)
    org = -T[:3, :3].T @ T[:3, 3]
    d = dc @ T[:3, :3]
    d = torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    far = torch.where(d > 0, (t64(room.size) - org) / d, -org / d)
    best, axis = far.min(1)
    surf = 2 * (2 - axis) + (torch.gather(d, 1, axis[:, None])[:, 0] > 0)
    for b, (lo, hi) in enumerate(room.boxes):
        t0, t1 = (t64(lo) - org) / d, (t64(hi) - org) / d
        tn, tf = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
        hit = (tn <= tf) & (tn > 1e-6) & (tn < best)
        best = torch.where(hit, tn, best)
        surf = torch.where(hit, 6 + b, surf)
    p = org + best[:, None] * d
    tex = 0.5 + 0.5 * torch.sin(7.0 * p[:, 0]) * torch.sin(5.0 * p[:, 1] + 3.0 * p[:, 2])
    rgb = (t64(room.albedo)[surf] * (0.6 + 0.4 * tex[:, None])).clamp(0, 1).T
    return best, rgb, torch.as_tensor(room.surface_class, device=DEV)[surf], p


def _cameras(case, seed):
    """The case's views: box scenes before an identity camera, others along the loop through the room."""
    w, h, fx, views = case["w"], case["h"], case.get("fx", float(case["w"])), case.get("views", 1)
    if case.get("scene") == "box":
        return [synth.camera(w, h, fx) for _ in range(views)]
    r = np.random.default_rng(seed)
    if case.get("scene") == "scan":  # consecutive frames
        poses = synth.smooth_path(views + 2, 0.6 + 0.01 * float(r.random()))[1:views + 1]
    else:
        poses = [synth.keyframe_loop()[i] for i in r.integers(0, 200, views)]
    cams = []
    for v, T in enumerate(poses):
        s = 640 / 1200 if case.get("ragged") and v % 2 else 1.0
        cams.append(synth.camera(max(16, round(w * s)), max(16, round(h * s)), fx * s, T_cw=T))
    return cams


def _field(case, seed, room):
    """The map's parameters as f32 tensors, with the benchmark's distributions (trained opacities for a scan)."""
    g, n, d = _gen(seed), case["n"], case.get("d", 0)
    rnd = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)
    nrm = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)
    mu, sd, logit, rgb = -4.0, 0.5, nrm(n), rnd(n, 3)
    if case["scene"] == "box":
        means = torch.stack([2 * rnd(n) - 1, 2 * rnd(n) - 1, 3 + 2 * rnd(n)], 1)
        mu, sd = -3.0, 0.3
    elif case["scene"] == "room":
        faces, _ = synth._room_faces(room)
        f = torch.as_tensor(np.array([np.concatenate(x) for x in faces]), device=DEV)
        area = torch.linalg.cross(f[:, 3:6], f[:, 6:9]).norm(dim=1)
        at = f[torch.searchsorted(torch.cumsum(area, 0) / area.sum(), rnd(n)).clamp(max=len(faces) - 1)]
        means = at[:, :3] + rnd(n, 1) * at[:, 3:6] + rnd(n, 1) * at[:, 6:9] + 0.01 * nrm(n, 3)
    else:
        # n pixels of three frames of the path, each Gaussian as wide as the spacing of its neighbours
        size = case["w"] * case["h"]
        parts, per = [], (n + 2) // 3
        for i, T in enumerate(synth.smooth_path(12, 2.0)[::4]):
            dep, col, _, p = _rays(room, synth.camera(case["w"], case["h"], case["fx"], T_cw=T))
            at = torch.randint(size, (min(per, n - i * per),), generator=g, device=DEV) if n > i * per else torch.zeros(0, dtype=torch.long, device=DEV)
            s = torch.log(dep[at] / case["fx"]) + 0.5 * math.log(max(1.0, size / n))
            parts.append((p[at], s, col[:, at].T))
        means, base, rgb = (torch.cat([q[j] for q in parts]) for j in range(3))
        means = means + 0.002 * nrm(n, 3)
        mu, sd, logit, rgb = base[:, None], 0.2, 1.5 + nrm(n), (rgb + 0.02 * nrm(n, 3)).clamp(0, 1)
    q = nrm(n, 4)
    out = dict(means=means, quats=q / q.norm(dim=1, keepdim=True), log_scales=mu + sd * nrm(n, 3), opacity_logits=logit,
               rgb=rgb, feat=nrm(n, d))
    out = {k: v.float().contiguous() for k, v in out.items()}
    if case.get("half"):
        out["rgb"], out["feat"] = out["rgb"].half(), out["feat"].bfloat16()
    return out


def _observe(case, cams, seed, room):
    """Colour, depth and label of every view, planar over all pixels, with the sensor's noise, holes and unlabelled pixels."""
    g, k = _gen(seed, 1), max(1, case.get("k", 8))
    dep, rgb, lab = (torch.cat(x, -1) for x in zip(*[_rays(room, c)[:3] for c in cams]))
    rnd = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)
    dep = dep * (1 + 0.002 * (rnd(dep.numel()) - 0.5))
    rgb = (rgb + 0.02 * (rnd(*rgb.shape) - 0.5)).clamp(0, 1)
    dep[rnd(dep.numel()).argsort()[:dep.numel() // 100]] = 0.0
    lab = torch.where(rnd(lab.numel()) < 0.01, torch.full_like(lab, 255), (lab * 3) % k)
    return dict(rgb=rgb.float().contiguous(), depth=dep.float().contiguous(), label=lab.to(torch.uint8).contiguous())


def _decoder(case, seed):
    g, s = _gen(seed, 2), 1.0 / math.sqrt(max(1, case["d"]))
    return (s * torch.randn(case["k"], case["d"], generator=g, device=DEV), s * torch.randn(case["k"], generator=g, device=DEV))


def _images(case, P, seed, tg):
    """What a render of a half-trained map looks like beside its observation (for the calls that start from images)."""
    g = _gen(seed, 3)
    rnd = lambda *s: torch.rand(*s, generator=g, device=DEV)
    seen = torch.ones(P, dtype=torch.bool, device=DEV)
    seen[(rnd(P) + 2.0 * (tg["depth"] <= 0)).argsort()[:round(case.get("unseen", 0.02) * P)]] = False
    sil = torch.where(seen, 1 - 0.012 * rnd(P), 0.4 * rnd(P))
    depth = sil * (torch.where(tg["depth"] > 0, tg["depth"], 2.0) * (1 + 0.04 * (rnd(P) - 0.5)))
    return dict(rgb=(tg["rgb"] + 0.2 * (rnd(3, P) - 0.5)), depth=depth, sil=sil,
                feat=torch.randn(max(case["d"], 1), P, generator=g, device=DEV))


def _adam_state(case, seed):
    """Parameters, gradients (zero for the four fifths of the map out of view) and moments of some earlier steps."""
    f, g, n = _field(dict(case, scene="room"), seed, synth.make_room()), _gen(seed, 4), case["n"]
    m = [1e-6 * torch.randn(n * (14 + case["d"]), generator=g, device=DEV),
         1e-12 * (0.01 + torch.rand(n * (14 + case["d"]), generator=g, device=DEV))]
    seen = torch.rand(n, generator=g, device=DEV) < 0.2
    grad = {k: 1e-6 * torch.randn(v.shape, generator=g, device=DEV) * (seen if v.dim() == 1 else seen[:, None]) for k, v in f.items()}
    return f, grad, torch.cat(m)


ADAM_STEPS = 25  # mapping iterations behind the adam case's moments


def _weights(case):
    return raster.LossWeights(ssim=case["ssim"])


def _track_start(cams):
    """The constant-velocity start: the true pose, off by a fraction of a degree and a centimetre."""
    return synth.perturb_pose(cams[0].T_cw, 0.4, 0.01)


def _inputs(case, seed):
    """Everything that a state is made of, without the framework's buffers."""
    room, kind = synth.make_room(int(seed) % 97), case["kind"]
    cams = _cameras(case, seed) if "w" in case else None
    x = dict(cams=cams, P=sum(c.width * c.height for c in cams) if cams else 0)
    if "scene" in case:
        x["field"] = _field(case, seed, room)
    if kind in ("step", "track", "loss", "expand"):
        x["targets"] = _observe(case, cams, seed, room)
    if kind in ("step", "track", "loss"):
        x["W"], x["b"] = _decoder(case, seed)
    if kind in ("loss", "expand"):
        x["images"] = _images(case, x["P"], seed, x["targets"])
    if kind == "autograd":
        g = _gen(seed, 5)
        x["grads"] = [torch.randn(s, generator=g, device=DEV) / x["P"] for s in ((3, x["P"]), (x["P"],), (x["P"],), (case["d"], x["P"]))]
    if kind == "expand":
        x["field"] = _field(dict(case, scene="room"), seed, room)
        x["feat_init"] = torch.randn(x["P"], case["d"], generator=_gen(seed, 6), device=DEV)
    return x


# ---------------------------------------------------------------------------------------- runs
def _warm_and_capture(fn):
    """Runs fn on a side stream (module loads), then captures it, as the framework's own loops do."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        fn()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fn()
    return graph


def prepare(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    st = dict(kind=kind, case=case)
    if kind == "adam":
        f, grad, m = _adam_state(case, seed)
        r = raster.Renderer(case["n"], [synth.camera(16, 16, 16.0)], case["d"], 1024)
        for name, k in zip(GROUPS, ("d_means", "d_quats", "d_log_scales", "d_logits", "d_rgb", "d_feat")):
            if name != "feat" or case["d"]:
                getattr(r, k).copy_(grad[name])
        field = raster.Field(**f)
        opt = raster.MappingAdam(field)
        opt.moments.copy_(m)
        opt.step_ctr.fill_(float(ADAM_STEPS))
        return dict(st, r=r, field=field, opt=opt)
    cams = x["cams"]
    if kind in ("loss", "expand"):
        r = raster.Renderer(0, cams, case["d"], 0, n_classes=case.get("k", 0))
        for name in ("rgb", "depth", "sil", "feat"):
            getattr(r, "img_" + name).copy_(x["images"][name])
        st.update(r=r, targets=x["targets"])
        if kind == "loss":
            w = raster.TRACKING if case["mask"] else raster.MAPPING
            return dict(st, W=x["W"], b=x["b"], w=w)
        return dict(st, field=raster.Field(**x["field"]), feat_init=x["feat_init"])
    field = raster.Field(**x["field"])
    d, k = case.get("d", 0), case.get("k", 0)
    if kind == "bin":  # room for four instances of every (view, Gaussian): the same for every seed
        r = raster.Renderer(field.n, cams, d, 4 * field.n * len(cams))
        r.forward(field)
        if r.status() != 0:
            raise RuntimeError("binning status %d" % r.status())
        r.vals.zero_()
        return dict(st, r=r, field=field)
    r = raster.fit_capacity(field, cams, d, margin=1.6 if kind == "track" else 1.25, n_classes=k)
    if kind == "track":
        tracker = raster.Tracker(field, cams[0], x["W"], x["b"], n_it=case["iters"], renderer=r)
        return dict(st, tracker=tracker, r=r, targets=x["targets"], T0=_track_start(cams))
    if kind == "autograd":
        leaves = [x["field"][g].requires_grad_() for g in GROUPS]
        return dict(st, r=r, leaves=leaves, grads=x["grads"])
    st.update(r=r, field=field)
    if kind == "step":
        mode = L.GS_GRAD_MAP | (L.GS_GRAD_POSE if case["pose"] else 0)
        st.update(targets=x["targets"], W=x["W"], b=x["b"])
        if case["scene"] == "scan" and case["views"] == 1:
            # the SLAM loop's keyframes: each iteration draws one and gathers its observation and pose
            store = slam.KeyframeStore(3, cams[0].width, cams[0].height)
            for s in range(3):
                store.rgb[s].copy_(x["targets"]["rgb"])
                store.depth[s].copy_(x["targets"]["depth"])
                store.label[s].copy_(x["targets"]["label"])
                store.put_pose(s, cams[0].T_cw)
            sampler = slam.RskmSampler(store, synth.rskm_draws(60, int(seed) % 1000))
            sampler.begin(0, 60, 3, 2, 2)

            def one():
                sampler.draw()
                r.iteration(field, sampler.targets, st["W"], st["b"], _weights(case), mode, pose_dev=sampler.pose)
            st["sampler"] = sampler
        else:
            def one():
                r.iteration(field, st["targets"], st["W"], st["b"], _weights(case), mode)
        st["graph"] = _warm_and_capture(one)
        st["graph"].replay()
        if r.status() != 0:
            raise RuntimeError("binning status %d" % r.status())
    return st


def run(st):
    kind, case, r = st["kind"], st["case"], st.get("r")
    if kind == "step":
        st["graph"].replay()
        # the loss and the twist are 64-bit sums of 32-bit terms: read as 32-bit values
        out = dict(means=r.d_means, quats=r.d_quats, log_scales=r.d_log_scales, opacity_logits=r.d_logits, rgb=r.d_rgb,
                   feat=r.d_feat, dec_W=r.d_dec_W, dec_b=r.d_dec_b, loss=r.loss_out.float(), img_rgb=r.img_rgb,
                   img_depth=r.img_depth, img_sil=r.img_sil)
        if case["pose"]:
            out["twist"] = r.d_twist.float()
        return out
    if kind == "track":
        T = st["tracker"].track(st["targets"], st["T0"])
        return dict(T=T.astype(np.float32), img_rgb=r.img_rgb, img_depth=r.img_depth, img_sil=r.img_sil)
    if kind == "render":
        r.forward(st["field"])
        return r.images()
    if kind == "autograd":
        outs = raster.rasterize(r, *st["leaves"])
        use = range(3 + (case["d"] > 0))
        want = st["leaves"][: 5 + (case["d"] > 0)]
        g = torch.autograd.grad([outs[i] for i in use], want, [st["grads"][i] for i in use])
        return dict(zip(GROUPS, g), **dict(zip(("img_rgb", "img_depth", "img_sil", "img_feat"), outs[: 3 + (case["d"] > 0)])))
    if kind == "bin":
        r.project(st["field"])
        r.bin_sort()
        return dict(uvdo=r.uvdo, conic=r.conic, touched=r.touched, vals=r.vals, ranges=r.ranges, n=r.n_inst)
    if kind == "loss":
        r.loss(st["targets"], st["W"], st["b"], st["w"])
        return dict(g_rgb=r.g_rgb, g_depth=r.g_depth, g_feat=r.g_feat, dec_W=r.d_dec_W, dec_b=r.d_dec_b,
                    loss=r.loss_out.float(), mask=r.mask, median=r.median)
    if kind == "adam":
        st["opt"].step(r)
        f = st["field"]
        return dict({k: getattr(f, k) for k in GROUPS[: 5 + (case["d"] > 0)]}, moments=st["opt"].moments)
    f, src, total, status = raster.expand(r, st["field"], st["targets"], st["feat_init"])
    return dict({k: getattr(f, k) for k in GROUPS[: 5 + (case["d"] > 0)]}, src=src, total=total, status=status)


# ---------------------------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; the blend's operations from the number of splats that
    a pixel blends before it saturates (about 75 on dense room surfaces, fewer on sparse ones)."""
    kind, n, d = case["kind"], case.get("n", 0), case.get("d", 0)
    cams = case.get("views", 1)
    P = 0
    if "w" in case:
        for v in range(cams):
            s = 640 / 1200 if case.get("ragged") and v % 2 and case.get("scene") != "box" else 1.0
            P += max(16, round(case["w"] * s)) * max(16, round(case["h"] * s))
    stored = 11 * 4 + (3 + d) * (2 if case.get("half") else 4)
    blend = min(75.0, 75.0 * n / 300_000) if case.get("scene") == "room" else 25.0
    image = (5 + d) * 4 * P
    fwd, bwd = P * blend * (24 + 2 * d), P * blend * (66 + 6 * d)
    if kind == "adam":
        return dict(bytes=28 * n * (14 + d), flops=12 * n * (14 + d))
    if kind == "loss":
        return dict(bytes=P * (17 + 4 * (5 + d) + 4 * (5 + d) + 4), flops=P * 6 * d * case["k"])
    if kind == "expand":
        new = case["unseen"] * P
        return dict(bytes=2 * 4 * (14 + d) * n + 12 * P + new * (12 + 4 * d + 4 * (14 + d) + 8), flops=20 * P)
    if kind == "bin":
        return dict(bytes=44 * n + 44 * n * cams, flops=300 * n * cams)
    if kind == "render":
        return dict(bytes=stored * n + image + 8 * P, flops=fwd + 300 * n)
    if kind == "autograd":
        return dict(bytes=stored * n + 2 * image + 4 * (14 + d) * n, flops=fwd + bwd + 800 * n)
    if kind == "track":
        it = case["iters"]  # the pose changes: every iteration reads the map again
        return dict(bytes=it * (stored * n + 17 * P), flops=it * (fwd + P * blend * 60 + 800 * n))
    return dict(bytes=stored * n + 17 * P + 4 * (14 + d) * n + 20 * P, flops=fwd + bwd + 800 * n * cams)


# ---------------------------------------------------------------- the method in 64 bits (torch)
TILE, ALPHA_MIN, ALPHA_MAX, T_MIN, Z_NEAR, LOWPASS = 16, 1.0 / 255.0, 0.99, 1e-4, 0.2, 0.3


def _hat(x):
    z = torch.zeros_like(x[0])
    return torch.stack([z, -x[5], x[4], x[0], x[5], z, -x[3], x[1], -x[4], x[3], z, x[2], z, z, z, z]).reshape(4, 4)


def _project(f, cam, T):
    """Centre, depth, opacity and conic (Eq. 2, 3) of every Gaussian; its tile rectangle (empty where culled) and depth key."""
    mu, R, t = f["means"], T[:3, :3], T[:3, 3]
    q = f["quats"] / f["quats"].norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                      1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                      1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    p = mu @ R.T + t
    pz = torch.where(p[:, 2] > Z_NEAR, p[:, 2], torch.ones_like(p[:, 2]))
    xz, yz = p[:, 0] / pz, p[:, 1] / pz
    W, H = cam.width, cam.height
    cx = xz.clamp((-cam.cx - 0.15 * W) / cam.fx, (W - cam.cx + 0.15 * W) / cam.fx)
    cy = yz.clamp((-cam.cy - 0.15 * H) / cam.fy, (H - cam.cy + 0.15 * H) / cam.fy)
    o = torch.zeros_like(pz)
    J = torch.stack([cam.fx / pz, o, -cam.fx * cx / pz, o, cam.fy / pz, -cam.fy * cy / pz], 1).view(-1, 2, 3)
    M = (J @ R) @ (Rq * f["log_scales"].exp()[:, None, :])
    S = M @ M.transpose(1, 2)
    a, b, c = S[:, 0, 0] + LOWPASS, S[:, 0, 1], S[:, 1, 1] + LOWPASS
    det = a * c - b * b
    u, v = cam.fx * xz + cam.cx, cam.fy * yz + cam.cy
    with torch.no_grad():
        ok = (p[:, 2] > Z_NEAR) & (det > 0)
        mid = 0.5 * (a + c)
        r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0))))
        TX, TY = (W + TILE - 1) // TILE, (H + TILE - 1) // TILE
        lim = lambda e, hi: e.clamp(-1e9, 1e9).long().clamp(0, hi)
        fl = lambda e: torch.floor(e / TILE)
        rect = torch.stack([lim(fl(u.floor() - r), TX), lim(fl(v.floor() - r), TY), lim(fl(u.floor() + r) + 1, TX),
                            lim(fl(v.floor() + r) + 1, TY)], 1) * ok[:, None]
        # the depth order is that of the 32-bit depths fma(r20, x, fma(r21, y, fma(r22, z, t_z)))
        key, r32 = t[2].float().double(), R[2].float().double()
        for i in (2, 1, 0):
            key = (r32[i] * mu[:, i] + key).float().double()
        rect = torch.cat([rect, key.float().view(torch.int32).long()[:, None]], 1)
    return dict(u=u, v=v, z=p[:, 2], o=torch.sigmoid(f["opacity_logits"]), A=c / det, B=-b / det, C=a / det), rect


@torch.no_grad()
def _tile_lists(s, rect, cam):
    """Chunks of (tile ids, [tiles, length] splat ids, -1 padded): each tile's splats by depth."""
    TX, TY = (cam.width + TILE - 1) // TILE, (cam.height + TILE - 1) // TILE
    n_touch = (rect[:, 2] - rect[:, 0]) * (rect[:, 3] - rect[:, 1])
    order = torch.argsort(rect[:, 4], stable=True)
    order = order[n_touch[order] > 0]
    k = n_touch[order]
    who = torch.repeat_interleave(order, k)
    j = torch.arange(who.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
    rw = rect[who, 2] - rect[who, 0]
    tile = (rect[who, 1] + j // rw) * TX + rect[who, 0] + j % rw
    tile, at = torch.sort(tile, stable=True)
    who = who[at]
    count = torch.bincount(tile, minlength=TX * TY)
    first = torch.cumsum(count, 0) - count
    chunks, big = [], torch.argsort(count, descending=True)
    sizes = count[big].tolist()
    i = 0
    while i < len(sizes):
        m = max(1, min(len(sizes) - i, 48_000_000 // (TILE * TILE * max(1, sizes[i]))))
        ids, ln = big[i:i + m], max(1, sizes[i])
        col = torch.arange(ln, device=DEV)
        idx = torch.where(col < count[ids][:, None], who[(first[ids][:, None] + col).clamp(max=max(0, who.numel() - 1))] if who.numel() else col * 0, -1)
        chunks.append((ids, idx))
        i += m
    return chunks


def _blend(s, x, cam, ids, idx):
    """Blended values x (with the depth and 1 behind them), transmittance and list position of the last splat (Eq. 4-7, 10)."""
    TX = (cam.width + TILE - 1) // TILE
    q = torch.arange(TILE * TILE, device=DEV)
    px = (ids % TX)[:, None] * TILE + q % TILE + 0.5
    py = (ids // TX)[:, None] * TILE + q // TILE + 0.5
    g = idx.clamp(min=0)
    at = lambda k: s[k][g][:, None, :]
    dx, dy = px[:, :, None] - at("u"), py[:, :, None] - at("v")
    pw = -0.5 * (at("A") * dx * dx + at("C") * dy * dy) - at("B") * dx * dy
    al = (at("o") * pw.exp()).clamp(max=ALPHA_MAX)
    al = torch.where((pw > 0) | (al < ALPHA_MIN) | (idx < 0)[:, None, :], 0.0, al)
    Ti = torch.exp(torch.cumsum(torch.log1p(-al), -1))
    keep = (Ti >= T_MIN) & (al > 0)
    w = torch.where(keep, al * (Ti / (1 - al)), 0.0)
    vals = torch.bmm(w, x[g])
    with torch.no_grad():
        T = torch.where(Ti >= T_MIN, Ti, 1.0).amin(-1)
        last = (keep * torch.arange(1, idx.shape[1] + 1, device=DEV)).amax(-1)
    return vals, T, last, px, py


def _render(s, rgb, feat, rect, cam, back=None):
    """Images [3 + 1 + 1 + D, P], T, n_contrib; with back (their gradient), the gradients of s, rgb and feat instead."""
    W, H, P, C = cam.width, cam.height, cam.width * cam.height, 5 + feat.shape[1]
    chunks = _tile_lists(s, rect, cam)
    leaf = {k: v.detach().requires_grad_(back is not None) for k, v in dict(s, rgb=rgb, feat=feat).items()}
    img = torch.zeros(C, P, dtype=torch.float64, device=DEV)
    T, last = torch.ones(P, dtype=torch.float64, device=DEV), torch.zeros(P, dtype=torch.long, device=DEV)
    for ids, idx in chunks:
        with torch.set_grad_enabled(back is not None):
            x = torch.cat([leaf["rgb"], leaf["z"][:, None], torch.ones_like(leaf["z"])[:, None], leaf["feat"]], 1)
            v, t, l, px, py = _blend(leaf, x, cam, ids, idx)
            inside = (px < W) & (py < H)
            pix = (py[inside].long() * W + px[inside].long())
            if back is None:
                img[:, pix], T[pix], last[pix] = v[inside].T, t[inside], l[inside]
            else:
                (v[inside] * back[:, pix].T).sum().backward()
    if back is None:
        return img, T, last
    return {k: v.grad if v.grad is not None else torch.zeros_like(v) for k, v in leaf.items()}


def _median(err):
    return torch.sort(err)[0][(err.numel() - 1) // 2] if err.numel() else torch.zeros((), device=DEV)


def _mask(sil, depth, dgt, w):
    err = (depth - dgt).abs()
    return (sil > w.tau_obs) & (dgt > 0) & (err < 10 * _median(err[dgt > 0])), _median(err[dgt > 0])


def _ssim(x, y):
    k = torch.arange(-5, 6, device=DEV, dtype=torch.float64)
    k = torch.exp(-k * k / (2 * 1.5 ** 2))
    k = k / k.sum()
    conv = lambda e: torch.nn.functional.conv2d(torch.nn.functional.conv2d(e[:, None], k.view(1, 1, 1, 11), padding=(0, 5)),
                                                k.view(1, 1, 11, 1), padding=(5, 0))[:, 0]
    mx, my = conv(x), conv(y)
    sx, sy, sxy = conv(x * x) - mx * mx, conv(y * y) - my * my, conv(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    return ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sx + sy + c2))).mean()


def _loss(img, tg, W, b, w, hw, m=None):
    """The loss terms of one view (Eq. 8, 15-17, 21): colour, depth, semantic."""
    rgb, depth, feat = img[:3], img[3], img[5:]
    P = depth.numel()
    m = torch.ones_like(depth) if m is None else m.double()
    l1 = (m * (rgb - tg["rgb"]).abs()).sum() / P
    if w.ssim:
        l1 = (1 - w.ssim) * l1 + w.ssim * (1 - _ssim(rgb.reshape(3, *hw), tg["rgb"].reshape(3, *hw)))
    ld = (m * (tg["depth"] > 0) * (depth - tg["depth"]).abs()).sum() / P
    z = W @ feat + b[:, None]
    on = tg["label"] < W.shape[0]
    ce = torch.logsumexp(z, 0) - torch.gather(z, 0, torch.where(on, tg["label"], 0)[None].long())[0]
    return torch.stack([w.color * l1, w.depth * ld, w.sem * (m * on * ce).sum() / P])


def _view(x, cams, v, key):
    a = sum(c.width * c.height for c in cams[:v])
    return x[key][..., a:a + cams[v].width * cams[v].height]


def _exact_step(case, x, w, tracked=None):
    """The gradients of one pass; tracked: a pose [4,4] to take instead of the camera's, for the twist alone."""
    cams = x["cams"]
    f = {k: v.double().requires_grad_(tracked is None) for k, v in x["field"].items()}
    W, b = (x[k].double().requires_grad_() for k in ("W", "b"))
    tg = {k: v.double() if v.dtype == torch.float32 else v for k, v in x["targets"].items()}
    terms, imgs, twists = 0.0, [], []
    for v, cam in enumerate(cams):
        xi = torch.zeros(6, dtype=torch.float64, device=DEV, requires_grad=True)
        T0 = torch.as_tensor(np.asarray(cam.T_cw), dtype=torch.float64, device=DEV) if tracked is None else tracked
        s, rect = _project(f, cam, (torch.eye(4, dtype=torch.float64, device=DEV) + _hat(xi)) @ T0)
        img, _, _ = _render(s, f["rgb"], f["feat"], rect, cam)
        img.requires_grad_()
        t = {k: _view(tg, cams, v, k) for k in tg}
        m = _mask(img[4].detach(), img[3].detach(), t["depth"], w)[0] if w.mask_mode else None
        ls = _loss(img, t, W, b, w, (cam.height, cam.width), m)
        ls.sum().backward()
        terms = terms + ls.detach()
        back = _render(s, f["rgb"], f["feat"], rect, cam, img.grad)
        outs = [(s[k], back[k]) for k in s] + ([(f[k], back[k]) for k in ("rgb", "feat")] if tracked is None else [])
        torch.autograd.backward([o for o, g in outs if o.requires_grad], [g for o, g in outs if o.requires_grad])
        imgs.append(img.detach())
        twists.append(xi.grad)
    img = torch.cat(imgs, 1)
    if tracked is not None:
        return img, twists[0]
    sc = f["log_scales"].detach().exp()
    mu, sd = sc.mean(), sc.std(unbiased=False)
    for on, lam, grad in ((sc > mu + 2 * sd, w.big, sc), (sc < mu - 2 * sd, w.small, -torch.ones_like(sc))):
        if on.any():
            f["log_scales"].grad += lam * on * grad / on.sum()
    out = {k: f[k].grad for k in GROUPS}
    out.update(dec_W=W.grad, dec_b=b.grad, loss=torch.cat([terms.sum()[None], terms]), img_rgb=img[:3], img_depth=img[3],
               img_sil=img[4])
    if case["pose"]:
        out["twist"] = torch.stack(twists)
    return out


def _exact_track(case, x):
    T = torch.as_tensor(_track_start(x["cams"]), dtype=torch.float64, device=DEV)
    m, v = torch.zeros(6, dtype=torch.float64, device=DEV), torch.zeros(6, dtype=torch.float64, device=DEV)
    lr = torch.as_tensor(raster.TRACKING_LR, dtype=torch.float64, device=DEV)
    for i in range(1, case["iters"] + 1):
        img, g = _exact_step(case, x, raster.TRACKING, tracked=T)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        T = torch.matrix_exp(_hat(-lr * (m / (1 - 0.9 ** i)) / ((v / (1 - 0.999 ** i)).sqrt() + 1e-15))) @ T
    return dict(T=T, img_rgb=img[:3], img_depth=img[3], img_sil=img[4])


def _exact_loss(case, x):
    cams, w = x["cams"], raster.TRACKING if case["mask"] else raster.MAPPING
    W, b = (x[k].double().requires_grad_() for k in ("W", "b"))
    im = x["images"]
    img = torch.cat([im["rgb"], im["depth"][None], im["sil"][None], im["feat"]]).double().requires_grad_()
    terms, masks, medians = 0.0, [], []
    for v, cam in enumerate(cams):
        t = {k: _view(x["targets"], cams, v, k) for k in x["targets"]}
        one = _view(dict(i=img), cams, v, "i")
        m, med = None, torch.zeros((), device=DEV)
        if case["mask"]:  # the mask is decided on the 32-bit values
            m, med = _mask(_view(im, cams, v, "sil"), _view(im, cams, v, "depth"), t["depth"], w)
        masks.append(torch.ones(cam.width * cam.height, dtype=torch.float64, device=DEV) if m is None else m.double())
        medians.append(med.double())
        t = {k: a.double() if a.dtype == torch.float32 else a for k, a in t.items()}
        terms = terms + _loss(one, t, W, b, w, (cam.height, cam.width), m)
    terms.sum().backward()
    return dict(g_rgb=img.grad[:3], g_depth=img.grad[3], g_feat=img.grad[5:], dec_W=W.grad, dec_b=b.grad,
                loss=torch.cat([terms.sum()[None], terms]).detach(), mask=torch.cat(masks), median=torch.stack(medians))


def _exact_adam(case, seed):
    f, grad, mom = _adam_state(case, seed)
    n, t, out, at = case["n"] * (14 + case["d"]), ADAM_STEPS + 1, {}, 0
    m, v = mom[:n].double(), mom[n:].double()
    for k, lr in zip(GROUPS, raster.MAPPING_LR):
        e = slice(at, at + f[k].numel())
        g = grad[k].double().reshape(-1)
        m[e], v[e] = 0.9 * m[e] + 0.1 * g, 0.999 * v[e] + 0.001 * g * g
        step = lr * (m[e] / (1 - 0.9 ** t)) / ((v[e] / (1 - 0.999 ** t)).sqrt() + 1e-15)
        out[k] = f[k].double() - step.reshape(f[k].shape)
        at = e.stop
    if not case["d"]:
        del out["feat"]
    return dict(out, moments=torch.cat([m, v]))


def _exact_expand(case, x):
    cam, tg, im = x["cams"][0], x["targets"], x["images"]
    dgt, err = tg["depth"], (im["depth"] - tg["depth"]).abs()
    un = (dgt > 0) & ((im["sil"] < 0.5) | ((im["depth"] > dgt) & (err > 50 * _median(err[dgt > 0]))))
    pix = un.nonzero()[:, 0]
    d, T = dgt[pix].double(), torch.as_tensor(cam.T_cw, dtype=torch.float64, device=DEV)
    pc = torch.stack([(pix % cam.width + 0.5 - cam.cx) / cam.fx * d, (pix // cam.width + 0.5 - cam.cy) / cam.fy * d, d], 1)
    k = pix.numel()
    new = dict(means=(pc - T[:3, 3]) @ T[:3, :3], quats=torch.eye(4, dtype=torch.float64, device=DEV)[:1].expand(k, 4),
               log_scales=torch.log(d / cam.fx)[:, None].expand(k, 3), opacity_logits=torch.zeros_like(d),
               rgb=tg["rgb"][:, pix].T.double(), feat=x["feat_init"][:k].double())
    out = {g: torch.cat([x["field"][g].double(), new[g]]) for g in GROUPS[: 5 + (case["d"] > 0)]}
    return dict(out, src=None, total=None, status=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "bin" or (kind == "track" and case["iters"] * case["w"] * case["h"] > 33_000_000):
        # whole numbers (and the records they are decided on); a long track of a large frame takes minutes
        return None
    if kind == "adam":
        return _exact_adam(case, seed)
    x = _inputs(case, seed)
    if kind == "loss":
        return _exact_loss(case, x)
    if kind == "expand":
        return _exact_expand(case, x)
    if kind == "track":
        return _exact_track(case, x)
    if kind == "step":
        return _exact_step(case, x, _weights(case))
    cam = x["cams"][0]
    T = torch.as_tensor(np.asarray(cam.T_cw), dtype=torch.float64, device=DEV)
    f = {k: v.double().requires_grad_(kind == "autograd") for k, v in x["field"].items()}
    s, rect = _project(f, cam, T)
    img, trans, last = _render(s, f["rgb"], f["feat"], rect, cam)
    if kind == "render":
        at = lambda e: e.view(*e.shape[:-1], cam.height, cam.width)
        return dict(rgb=at(img[:3]), depth=at(img[3]), sil=at(img[4]), feat=at(img[5:]), T=at(trans), n_contrib=None)
    g = x["grads"]
    back = _render(s, f["rgb"], f["feat"], rect, cam, torch.cat([g[0], g[1][None], g[2][None], g[3]]).double())
    torch.autograd.backward([s[k] for k in s] + [f["rgb"]] + ([f["feat"]] if case["d"] else []),
                            [back[k] for k in s] + [back["rgb"]] + ([back["feat"]] if case["d"] else []))
    use = 3 + (case["d"] > 0)
    return dict({k: f[k].grad for k in GROUPS[: 5 + (case["d"] > 0)]},
                **dict(zip(("img_rgb", "img_depth", "img_sil", "img_feat"), (img[:3], img[3], img[4], img[5:])[:use])))
