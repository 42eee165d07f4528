"""Performance cases of the Gaussian-map optimiser: what a mapping program has it do.

A case is a dict of plain values.  Five kinds of work, each through the public Python binding:

  step    ``Map.optimize_step`` on one keyframe or a window of keyframes, and the updated Gaussians read back
          on the device (forward, exposure, L1 + D-SSIM, backward, fused Adam)
  grad    the differentiable path: ``autograd.render`` + ``autograd.photometric_loss`` and the gradients of every
          Gaussian attribute, of the pose twist and of the exposure, with upstream depth and opacity gradients
  render  ``Map.render`` of a novel view (colour, depth, opacity) into device memory
  loss    the photometric loss alone, with its gradients, through either entry point
  expand  a keyframe's points offered to a map through its opacity mask (``Map.add_points``)

Two scenes: ``frustum`` (random Gaussians in one camera's frustum, the small and the differentiation workloads) and
``street`` (LiDAR sweeps along a road between box facades plus a sky hemisphere, the outdoor workload), both drawn
from the seed alone.  A street map is jittered around its initialisation (anisotropic scales, spread opacities,
non-zero higher SH bands), as it is while it is being optimised.

``exact`` renders, differentiates and updates in 64 bits with plain torch.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2404_06926_gb300 import autograd as ag
from paper_2404_06926_gb300 import binding, scenes

DEV = "cuda"
LR = dict(means=1.6e-4, log_scales=5e-3, quats=1e-3, logits=0.05, dc=2.5e-3, rest=2.5e-3 / 20.0, exposure=1e-3)
# The optimiser's usual epsilon.  (The map's default, 1e-15, makes the first update of every element the sign of its
# gradient, rounding noise included; the work of a step is the same.)
EPS = 1e-8
NAMES = ("means", "log_scales", "quats", "logits", "sh")


# ---------------------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------------------
def _step(**kw):
    c = dict(kind="step", scene="street", n=250_000, deg=3, width=640, height=512, views=1, mixed=False, tuned=True,
             repro=False, sparse=True, host_image=False)
    c.update(kw)
    return c


def _grad(**kw):
    c = dict(kind="grad", scene="street", n=250_000, deg=3, width=640, height=480, tile=16, extras=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest map: 2,000 Gaussians without view-dependent colour in a 128 x 96 view, default execution;
        # launches and host work count
        _step(name="step_2k_128x96", scene="frustum", n=2_000, deg=0, width=128, height=96, tuned=False),
        # one optimisation step at a LiDAR-camera rig's frame size, graph replay: the mapping thread's inner loop
        _step(name="step_250k_640x512"),
        # the outdoor map at full size
        _step(name="step_1m_1280x1024", n=1_000_000, width=1280, height=1024),
        # an odd frame size, degree 2, every Gaussian updated (dense Adam), default execution, frames from pinned host memory
        _step(name="step_300k_957x717_dense", n=300_000, deg=2, width=957, height=717, tuned=False, sparse=False,
              host_image=True),
        # bit-reproducible steps (fixed summation order)
        _step(name="step_250k_640x512_repro", repro=True),
        # the batched form: a window of 12 keyframes of three resolutions over 2M Gaussians, the largest call
        _step(name="window12_2m_mixed", n=2_000_000, width=1280, height=1024, views=12, mixed=True),
        # the differentiation check: 5,000 Gaussians, 256 x 192, pose and exposure gradients
        _grad(name="grad_5k_256x192", scene="frustum", n=5_000, width=256, height=192, extras=False),
        # the same on a street view, with gradients through the depth and opacity images (pose refinement against LiDAR depth)
        _grad(name="grad_250k_640x480"),
        # a served novel view at the largest requested size
        dict(name="render_1m_1920x1080", kind="render", scene="street", n=1_000_000, deg=3, width=1920, height=1080,
             tuned=True),
        # the loss alone on a full-size frame, and on a ragged one through the entry point that allocates nothing
        dict(name="loss_1280x1024", kind="loss", width=1280, height=1024, noalloc=False),
        dict(name="loss_647x481_noalloc", kind="loss", width=647, height=481, noalloc=True),
        # a keyframe's LiDAR and visual points offered to a map of half a million Gaussians
        dict(name="expand_60k_into_500k", kind="expand", scene="street", n=500_000, deg=3, width=640, height=512,
             points=60_000),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame(rng, lo, hi):
    """A frame of lo..hi pixels (log-uniform), aspect 1.2 to 1.8, any parity."""
    p, a = math.exp(rng.uniform(math.log(lo), math.log(hi))), rng.uniform(1.2, 1.8)
    return int(round(math.sqrt(p * a))), int(round(math.sqrt(p / a)))


def draw(rng):
    kind = rng.choice(("step", "step", "grad", "render", "loss", "expand"))
    if kind == "loss":
        w, h = _frame(rng, 20_000, 2_000_000)
        return dict(kind="loss", width=w, height=h, noalloc=rng.random() < 0.3)
    if kind == "expand":
        w, h = _frame(rng, 100_000, 1_400_000)
        return dict(kind="expand", scene="street", n=_logint(rng, 50_000, 1_000_000), deg=3, width=w, height=h,
                    points=_logint(rng, 5_000, 100_000))
    if kind == "render":
        w, h = _frame(rng, 100_000, 2_100_000)
        return dict(kind="render", scene="street", n=_logint(rng, 30_000, 1_200_000), deg=rng.randint(0, 3), width=w,
                    height=h, tuned=rng.random() < 0.7)
    if rng.random() < 0.25:
        n = _logint(rng, 1_000, 8_000)
        w, h = _frame(rng, 10_000, 60_000)
        if kind == "grad":
            return _grad(scene="frustum", n=n, deg=rng.randint(0, 3), width=w, height=h, tile=rng.choice((8, 16, 32)),
                         extras=rng.random() < 0.5)
        return _step(scene="frustum", n=n, deg=rng.randint(0, 3), width=w, height=h, tuned=rng.random() < 0.5)
    n = _logint(rng, 20_000, 1_200_000)
    w, h = _frame(rng, 100_000, 1_400_000)
    if kind == "grad":
        return _grad(n=n, deg=rng.randint(0, 3), width=w, height=h, tile=rng.choice((8, 16, 16, 32)),
                     extras=rng.random() < 0.5)
    views = rng.choice((1, 1, 1, 2, 4))
    return _step(n=n, deg=rng.choice((1, 2, 3, 3, 3)), width=w, height=h, views=views, mixed=views > 1 and rng.random() < 0.6,
                 tuned=rng.random() < 0.7, repro=rng.random() < 0.15, sparse=rng.random() < 0.8,
                 host_image=rng.random() < 0.3)


# ---------------------------------------------------------------------------------------------------------------
# inputs (plain torch; the street's geometry and trajectory are the package's seeded scene generator)
# ---------------------------------------------------------------------------------------------------------------
def _f32(x):
    return torch.as_tensor(np.asarray(x), dtype=torch.float32, device=DEV)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _cast(sc, o, d):
    """Nearest hit of the rays o + s d with the street's ground and boxes: (s, colour), s = inf where there is none."""
    s = -o[:, 2] / d[:, 2]
    hx, hy = o[:, 0] + s * d[:, 0], o[:, 1] + s * d[:, 1]
    ok = (s > 0) & torch.isfinite(s) & (hx > -20) & (hx < 420) & (hy.abs() < 60)
    best = torch.where(ok, s, torch.full_like(s, math.inf))
    tex = 0.75 + 0.25 * torch.remainder(torch.floor(hx / 2) + torch.floor(hy / 2), 2)
    col = _f32(sc.ground_col)[None] * tex[:, None]
    inv = 1.0 / torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    lo, hi = _f32(sc.box_lo), _f32(sc.box_hi)
    for b in range(lo.shape[0]):
        t0, t1 = (lo[b] - o) * inv, (hi[b] - o) * inv
        tmin, tmax = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
        hit = (tmax >= tmin) & (tmin > 0) & (tmin < best)
        p = o + torch.where(hit, tmin, torch.zeros_like(tmin))[:, None] * d
        fr = float(sc.box_freq[b])
        pat = 0.7 + 0.3 * torch.remainder(torch.floor(p[:, 0] * fr) + torch.floor(p[:, 1] * fr) + torch.floor(p[:, 2] * fr * 0.7), 2)
        best = torch.where(hit, tmin, best)
        col = torch.where(hit[:, None], _f32(sc.box_col[b])[None] * pat[:, None], col)
    return best, col


def _street_points(sc, g, n, poses, width, height, f):
    """n coloured points (LiDAR, and 5% visual points above its top beam) in capture order: (xyz, rgb, depth)."""
    R = _f32(np.stack([sc.pose(float(s))[0] for s in poses]))
    t = _f32(np.stack([sc.pose(float(s))[1] for s in poses]))
    half, parts, have = math.atan(width / 2 / f), [], 0
    while have < n:
        m = int(1.6 * (n - have)) + 1024
        k = torch.randint(len(poses), (m,), generator=g, device=DEV)
        el = (torch.randint(32, (m,), generator=g, device=DEV).float() * (30.0 / 31) - 15.0) * (math.pi / 180)
        az = (_rand(g, m) * 2 - 1) * half
        lidar = torch.stack([torch.sin(az) * torch.cos(el), -torch.sin(el), torch.cos(az) * torch.cos(el)], 1)
        u, v = _rand(g, m) * width, _rand(g, m) * height * 0.45
        visual = torch.stack([(u - width / 2) / f, (v - height / 2) / f, torch.ones_like(u)], 1)
        visual = visual / visual.norm(dim=1, keepdim=True)
        is_vis = _rand(g, m) < 0.12
        dc = torch.where(is_vis[:, None], visual, lidar)
        Rk, tk = R[k], t[k]
        d = torch.einsum("mij,mi->mj", Rk, dc)
        o = -torch.einsum("mij,mi->mj", Rk, tk)
        s, col = _cast(sc, o, d)
        s = s + 0.02 * _randn(g, m)
        p = o + torch.where(torch.isfinite(s), s, torch.zeros_like(s))[:, None] * d
        pc = torch.einsum("mij,mj->mi", Rk, p) + tk
        uu, vv = f * pc[:, 0] / pc[:, 2] + width / 2, f * pc[:, 1] / pc[:, 2] + height / 2
        ok = torch.isfinite(s) & (pc[:, 2] > 0.5) & (uu >= 0) & (uu < width) & (vv >= 0) & (vv < height)
        ok &= ~is_vis | (p[:, 2] > sc.cam_h + 1.0)
        parts.append((k[ok], p[ok], col[ok], pc[ok, 2]))
        have += int(ok.sum())
    k, p, col, z = (torch.cat(x)[:n] for x in zip(*parts))
    order = torch.sort(k, stable=True).indices
    return p[order].contiguous(), col[order].contiguous(), z[order].contiguous()


def _street(case, seed):
    """The scene, its cameras and a jittered map of case['n'] Gaussians, a tenth of them sky."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    W, H = case["width"], case["height"]
    f = 0.78125 * W
    sc = scenes.Outdoor(seed=seed, width=W, img_height=H, f=f)
    n_sky = case["n"] // 10
    n, K = case["n"] - n_sky, (case["deg"] + 1) ** 2
    p, col, z = _street_points(sc, g, n, sc.traj_x, W, H, f)
    # sky: uniform by area on the upper hemisphere of radius 1e4, scale about the nearest neighbour's distance
    zc, ph = _rand(g, n_sky), 2 * math.pi * _rand(g, n_sky)
    rr = (1 - zc * zc).clamp_min(0).sqrt()
    sky = 1e4 * torch.stack([rr * torch.cos(ph), rr * torch.sin(ph), zc], 1)
    ls = torch.cat([torch.log(z / f), torch.full((n_sky,), math.log(0.5e4 * math.sqrt(2 * math.pi / max(n_sky, 1))), device=DEV)])
    lg = torch.cat([torch.full((n,), math.log(0.1 / 0.9), device=DEV), torch.full((n_sky,), math.log(0.7 / 0.3), device=DEV)])
    dc = (torch.cat([col, torch.ones_like(sky)]) - 0.5) / 0.28209479177387814
    N = n + n_sky
    q = 0.3 * _randn(g, N, 4)
    q[:, 0] += 1.0
    sh = torch.zeros(N, K, 3, device=DEV)
    sh[:, 0] = dc + 0.1 * _randn(g, N, 3)
    if K > 1:
        sh[:, 1:] = 0.05 * _randn(g, N, K - 1, 3)
    params = dict(means=torch.cat([p, sky]).contiguous(), log_scales=(ls[:, None] + 0.15 + 0.3 * _randn(g, N, 3)).contiguous(),
                  quats=q.contiguous(), logits=(lg + 1.0 + 1.2 * _randn(g, N)).contiguous(), sh=sh.contiguous())
    sizes = [(W, H)] if not case.get("mixed") else [(W, H), (max(8, W * 4 // 5), max(8, H * 3 // 4)), (max(8, W // 2), max(8, H // 2))]
    count = max(4, case.get("views", 1))
    pos = np.linspace(sc.traj_x[2], sc.traj_x[-12], count) + 0.37
    cams = [sc.camera_at(float(s), width=sizes[i % len(sizes)][0], height=sizes[i % len(sizes)][1], f=0.78125 * sizes[i % len(sizes)][0])
            for i, s in enumerate(pos)]
    return sc, g, params, cams


def _street_targets(sc, cams, seed):
    rng = np.random.default_rng(seed + 77)
    return [sc.target_image_torch(cam, device=DEV, rng=rng) for cam in cams]


def _frustum(case, seed):
    """Random Gaussians uniform in the frustum of one camera; uniform random targets."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    W, H, n, K = case["width"], case["height"], case["n"], (case["deg"] + 1) ** 2
    cam = scenes.camera(W, H, 100.0 * W / 128, 100.0 * W / 128, W / 2, H / 2)
    z = 0.5 + 9.5 * _rand(g, n)
    xy = torch.stack([(_rand(g, n) * W - cam["cx"]) * z / cam["fx"], (_rand(g, n) * H - cam["cy"]) * z / cam["fy"], z], 1)
    q = _randn(g, n, 4)
    params = dict(means=xy.contiguous(), log_scales=-2.0 + 0.5 * _randn(g, n, 3), quats=(q / q.norm(dim=1, keepdim=True)).contiguous(),
                  logits=_randn(g, n), sh=(0.5 if K == 1 else 0.2) * _randn(g, n, K, 3))
    return g, params, [cam], [_rand(g, H, W, 3)]


def _scene(case, seed, targets=True):
    """(params, cams, targets, sc, generator)"""
    if case["scene"] == "frustum":
        g, params, cams, imgs = _frustum(case, seed)
        return params, cams, imgs, None, g
    sc, g, params, cams = _street(case, seed)
    return params, cams, _street_targets(sc, cams, seed) if targets else None, sc, g


def _windows(case, cams):
    """Index lists of the keyframes that successive steps use."""
    v = case["views"]
    return [list(range(v))] if v > 1 else [[i] for i in range(len(cams))]


def _loss_inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    W, H = case["width"], case["height"]
    sc = scenes.Outdoor(seed=seed, width=W, img_height=H, f=0.78125 * W)
    tgt = sc.target_image_torch(sc.camera_at(30.0), device=DEV, rng=np.random.default_rng(seed))
    rgb = (tgt + 0.08 * _randn(g, H, W, 3)).clamp(0, 1.2).contiguous()
    E = torch.cat([torch.eye(3, device=DEV), torch.zeros(3, 1, device=DEV)], 1) + 0.03 * _randn(g, 3, 4)
    return rgb, tgt, E.contiguous()


def _grad_inputs(case, seed):
    params, cams, imgs, _, g = _scene(case, seed)
    H, W = case["height"], case["width"]
    twist = torch.tensor([0.02, -0.01, 0.03, 0.004, -0.006, 0.005], device=DEV)
    E = torch.cat([torch.eye(3, device=DEV), torch.zeros(3, 1, device=DEV)], 1) + 0.02 * _randn(g, 3, 4)
    gD = gO = None
    if case["extras"]:
        gD, gO = 1e-7 * _randn(g, H, W), 1e-6 * _randn(g, H, W)
    return params, cams[0], imgs[0], twist, E.contiguous(), gD, gO


def _expand_inputs(case, seed):
    sc, g, params, _ = _street(case, seed)
    pos = float(sc.traj_x[35]) + 0.5   # between two of the poses that the map was captured from
    cam = sc.camera_at(pos)
    xyz, rgb, _ = _street_points(sc, g, case["points"], [pos], case["width"], case["height"], cam["fx"])
    return params, cam, xyz, rgb


# ---------------------------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------------------------------------------
def _make_map(case, params, room=0):
    n = int(params["means"].shape[0])
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=case["deg"], capacity_hint=n + room, adam_eps=EPS,
                                           sparse_adam=1 if case.get("sparse", True) else 0))
    m.set_params(params)
    if case.get("tuned"):   # what the autotuner picks for steps on these scenes
        m.set_exec(use_graphs=1, persistent=1, segment=512)
    if case.get("repro"):
        m.set_exec(deterministic=1)
    return m


def _read_params(m, out):
    """The map's Gaussians into device tensors (at least as many rows as the map has)."""
    gs = binding.gaussians(out)
    binding.check(binding.lib().gl_map_get_params(m._h, ctypes.byref(gs), None))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss":
        rgb, tgt, E = _loss_inputs(case, seed)
        return dict(kind=kind, rgb=rgb, tgt=tgt, E=E, noalloc=case["noalloc"], ctx=binding.Ctx())
    if kind == "grad":
        params, cam, img, twist, E, gD, gO = _grad_inputs(case, seed)
        return dict(kind=kind, params={k: v.requires_grad_() for k, v in params.items()}, cam=cam, img=img,
                    twist=twist.requires_grad_(), E=E.requires_grad_(), gD=gD, gO=gO, tile=case["tile"], ctx=binding.Ctx())
    if kind == "render":
        params, cams, _, _, _ = _scene(case, seed, targets=False)
        H, W = case["height"], case["width"]
        out = (torch.empty(H, W, 3, device=DEV), torch.empty(H, W, device=DEV), torch.empty(H, W, device=DEV))
        return dict(kind=kind, map=_make_map(case, params), cams=cams, out=out, i=0)
    if kind == "expand":
        params, cam, xyz, rgb = _expand_inputs(case, seed)
        room = case["points"]
        out = {k: torch.zeros((v.shape[0] + room,) + tuple(v.shape[1:]), device=DEV) for k, v in params.items()}
        return dict(kind=kind, map=_make_map(case, params, room), params=params, cam=cam, xyz=xyz, rgb=rgb, out=out)
    params, cams, imgs, _, _ = _scene(case, seed)
    m = _make_map(case, params)
    images = [None] * len(cams)
    for k, (cam, img) in enumerate(zip(cams, imgs)):
        m.add_keyframe(k, cam, img)
    if case["host_image"]:
        images = [img.cpu().pin_memory() for img in imgs]
    windows = [[(k, cams[k], images[k]) for k in w] for w in _windows(case, cams)]
    return dict(kind=kind, map=m, windows=windows, out={k: torch.empty_like(v) for k, v in params.items()}, i=0)


def run(state):
    kind = state["kind"]
    if kind == "step":
        m, views = state["map"], state["windows"][state["i"] % len(state["windows"])]
        state["i"] += 1
        loss = m.optimize_step(views, want_loss=True)
        _read_params(m, state["out"])
        return dict(loss=loss, exposure=[m.exposure(v[0]) for v in views], params=state["out"])
    if kind == "grad":
        p, gD, gO = state["params"], state["gD"], state["gO"]
        rgb, depth, opac = ag.render(p, state["cam"], state["twist"], tile=state["tile"], glctx=state["ctx"])
        loss = ag.photometric_loss(rgb, state["img"], state["E"], glctx=state["ctx"])
        ins = [p[k] for k in NAMES] + [state["twist"], state["E"]]
        if gD is None:
            grads = torch.autograd.grad(loss, ins)
        else:
            grads = torch.autograd.grad([loss, depth, opac], ins, [None, gD, gO])
        return dict(rgb=rgb.detach(), depth=depth.detach(), opacity=opac.detach(), loss=loss.detach(), grads=list(grads))
    if kind == "render":
        rgb, depth, opac = state["out"]
        cam = state["cams"][state["i"] % len(state["cams"])]
        state["i"] += 1
        state["map"].render(cam, out_rgb=rgb, out_depth=depth, out_opacity=opac)
        return dict(rgb=rgb, depth=depth, opacity=opac)
    if kind == "loss":
        if state["noalloc"]:
            loss, dC, dE = binding.photometric_loss_noalloc(state["rgb"], state["tgt"], state["E"])
        else:
            loss, dC, dE = state["ctx"].loss(state["rgb"], state["tgt"], state["E"])
        return dict(loss=loss, dC=dC, dE=dE)
    # expand: the same map each time, then the keyframe's points
    m, out = state["map"], state["out"]
    m.set_params(state["params"])
    added = m.add_points(state["xyz"], state["rgb"], state["cam"], use_mask=True)
    _read_params(m, out)
    return dict(added=added, params=out)   # the rows past the map's end stay zero


# ---------------------------------------------------------------------------------------------------------------
# what one pass cannot do without (each input read once, each output written once; the pixels' blends by typical counts)
# ---------------------------------------------------------------------------------------------------------------
def _pixels(case):
    p = case["width"] * case["height"]
    if case["kind"] == "step":
        v = case["views"]
        if case["mixed"]:
            return sum(p if i % 3 == 0 else p * 3 // 5 if i % 3 == 1 else p // 4 for i in range(v))
        return p * v
    return p


def work(case):
    kind, P = case["kind"], _pixels(case)
    if kind == "loss":
        return dict(bytes=36.0 * P, flops=3 * 270.0 * P)   # colour, target, gradient; 5 + 3 separable 11-tap blurs
    n, row = case["n"], 44.0 + 12.0 * (case["deg"] + 1) ** 2
    blends = (40.0 if case["scene"] == "street" else 60.0) * P   # (pixel, Gaussian) pairs blended
    seen = 0.55 * n if case["scene"] == "street" else 0.95 * n    # Gaussians a view reaches
    if kind == "render":
        return dict(bytes=12.0 * n + seen * row + 20.0 * P, flops=22 * blends)
    if kind == "expand":   # the map is written once more, the points once
        return dict(bytes=(12.0 * n + seen * row) + 2 * n * row + n * 2 * row + case["points"] * (24.0 + row), flops=22 * blends)
    if kind == "grad":
        return dict(bytes=12.0 * n + seen * row + n * row + 72.0 * P, flops=85 * blends + 810.0 * P)
    moved = seen if case["sparse"] else float(n)
    return dict(bytes=12.0 * n * case["views"] + moved * row * 6 + 24.0 * P + 2 * n * row, flops=85 * blends + 810.0 * P)


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------------------------------------------
def _sh_basis(d, K):
    x, y, z = d.unbind(1)
    c0, c1 = 0.5 * math.sqrt(1 / math.pi), math.sqrt(3 / (4 * math.pi))
    Y = [torch.full_like(x, c0)]
    if K > 1:
        Y += [-c1 * y, c1 * z, -c1 * x]
    xx, yy, zz = x * x, y * y, z * z
    if K > 4:
        a, b = 0.5 * math.sqrt(15 / math.pi), 0.25 * math.sqrt(5 / math.pi)
        Y += [a * x * y, -a * y * z, b * (2 * zz - xx - yy), -a * x * z, 0.5 * a * (xx - yy)]
    if K > 9:
        a, b = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi)
        c, e = 0.25 * math.sqrt(21 / (2 * math.pi)), 0.25 * math.sqrt(7 / math.pi)
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy), e * z * (2 * zz - 3 * xx - 3 * yy),
              -c * x * (4 * zz - xx - yy), 0.5 * b * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return torch.stack(Y, 1)


class _Exact:
    """One view of a map in 64 bits: projection (differentiable), tile lists, blending by chunks of tiles."""

    PAIRS = 24_000_000   # (pixel, Gaussian) pairs of a chunk

    def __init__(self, params, cam, tile, twist=None):
        """params: 64-bit tensors (leaves where gradients are wanted); twist: 6 numbers or None."""
        self.W, self.H, self.Ts = cam["width"], cam["height"], tile
        f64 = dict(dtype=torch.float64, device=DEV)
        R, t = torch.tensor(np.asarray(cam["R"]), **f64), torch.tensor(np.asarray(cam["t"]), **f64)
        if twist is not None:
            rho, phi = twist[:3], twist[3:]
            o = torch.zeros((), **f64)
            A = torch.stack([torch.stack([o, -phi[2], phi[1], rho[0]]), torch.stack([phi[2], o, -phi[0], rho[1]]),
                             torch.stack([-phi[1], phi[0], o, rho[2]]), torch.stack([o, o, o, o])])
            G = torch.linalg.matrix_exp(A)
            R, t = G[:3, :3] @ R, G[:3, :3] @ t + G[:3, 3]
        mu, fx, fy, cx, cy = params["means"], cam["fx"], cam["fy"], cam["cx"], cam["cy"]
        pc = mu @ R.T + t
        x, y, z = pc.unbind(1)
        front = z.detach() > 0.2
        zs = torch.where(front, z, torch.ones_like(z))
        u, v = fx * x / zs + cx, fy * y / zs + cy
        q = params["quats"] / params["quats"].norm(dim=1, keepdim=True)
        w, a, b, c = q.unbind(1)
        Rq = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                          2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                          2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).view(-1, 3, 3)
        M = Rq * torch.exp(params["log_scales"])[:, None, :]
        lx, ly = 1.3 * 0.5 * self.W / fx, 1.3 * 0.5 * self.H / fy
        xz, yz = (x / zs).clamp(-lx, lx), (y / zs).clamp(-ly, ly)
        o = torch.zeros_like(zs)
        J = torch.stack([fx / zs, o, -fx * xz / zs, o, fy / zs, -fy * yz / zs], 1).view(-1, 2, 3)
        TM = torch.bmm(J @ R, M)
        S = torch.bmm(TM, TM.transpose(1, 2))
        sa, sb, sc = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
        det = sa * sc - sb * sb
        mid = 0.5 * (sa + sc)
        lam = mid + torch.sqrt(torch.clamp(mid * mid - det, min=0.1))
        with torch.no_grad():
            r = torch.ceil(3 * torch.sqrt(lam))
            TX, TY = -(-self.W // tile), -(-self.H // tile)
            x0, x1 = (torch.floor((u - r) / tile).clamp(0, TX), torch.floor((u + r + tile - 1) / tile).clamp(0, TX))
            y0, y1 = (torch.floor((v - r) / tile).clamp(0, TY), torch.floor((v + r + tile - 1) / tile).clamp(0, TY))
            area = ((x1 - x0) * (y1 - y0)).long()
            area = torch.where(front & (det > 0), area, torch.zeros_like(area))
            self.visible = area > 0
            ids = self.visible.nonzero()[:, 0]
            # ties of the depth order are those of 32-bit depths
            Rf, tf, mf = R.float(), t.float(), mu.detach().float()
            zf = Rf[2, 0] * mf[:, 0] + Rf[2, 1] * mf[:, 1] + Rf[2, 2] * mf[:, 2] + tf[2]
            ids = ids[torch.sort(zf[ids], stable=True).indices]
            cnt = area[ids]
            own = torch.repeat_interleave(ids, cnt)
            k = torch.arange(own.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            wd = (x1 - x0).long()[own]
            tiles = (y0.long()[own] + k // wd) * TX + x0.long()[own] + k % wd
            order = torch.sort(tiles, stable=True).indices
            self.own, self.count = own[order], torch.bincount(tiles, minlength=TX * TY)
            self.first = torch.cumsum(self.count, 0) - self.count
            self.TX = TX
        cw = -(R.T @ t)
        d = mu - cw
        Y = _sh_basis(d / d.norm(dim=1, keepdim=True), params["sh"].shape[1])
        rgb = torch.clamp((Y[:, :, None] * params["sh"]).sum(1) + 0.5, min=0.0)
        ok = torch.where(det > 0, det, torch.ones_like(det))
        # per Gaussian: u, v, conic A B C, opacity, r, g, b, depth
        self.feat = torch.stack([u, v, sc / ok, -sb / ok, sa / ok, torch.sigmoid(params["logits"]), rgb[:, 0], rgb[:, 1], rgb[:, 2], z], 1)

    def chunks(self):
        """Groups of tiles of about equal list length."""
        cnt = self.count.cpu().numpy()
        order = np.argsort(-cnt, kind="stable")
        order = order[cnt[order] > 0]
        i = 0
        while i < len(order):
            L = int(cnt[order[i]])
            k = max(1, int(self.PAIRS // (L * self.Ts * self.Ts)))
            yield torch.as_tensor(order[i:i + k].copy(), device=DEV), L
            i += k

    def blend(self, feat, tiles, L):
        """Colour, depth and opacity (5 values) of the tiles' pixels, and where they go in the image."""
        Ts = self.Ts
        j = torch.arange(L, device=DEV)[None]
        has = j < self.count[tiles][:, None]
        idx = self.own[torch.where(has, self.first[tiles][:, None] + j, torch.zeros_like(j))]
        F = feat[idx]                                       # B x L x 10
        pp = torch.arange(Ts * Ts, device=DEV)
        px, py = (tiles % self.TX * Ts)[:, None] + pp % Ts, (tiles // self.TX * Ts)[:, None] + pp // Ts   # B x P
        dx, dy = F[:, :, None, 0] - px[:, None, :], F[:, :, None, 1] - py[:, None, :]
        power = -0.5 * (F[:, :, None, 2] * dx * dx + F[:, :, None, 4] * dy * dy) - F[:, :, None, 3] * dx * dy
        alpha = torch.clamp(F[:, :, None, 5] * torch.exp(power), max=0.99)
        live = has[:, :, None] & (power <= 0) & (alpha >= 1 / 255)
        alpha = torch.where(live, alpha, torch.zeros_like(alpha))
        lt = torch.log1p(-alpha)
        run_ = torch.cumsum(lt, 1)
        wgt = alpha * torch.exp(run_ - lt) * (run_.detach() >= math.log(1e-4))
        val = torch.cat([F[:, :, 6:10], torch.ones_like(F[:, :, :1])], 2)   # r, g, b, depth, 1
        out = torch.bmm(wgt.transpose(1, 2), val)           # B x P x 5
        inside = (px < self.W) & (py < self.H)
        return out[inside], (py * self.W + px)[inside]

    def image(self):
        img = torch.zeros(self.H * self.W, 5, dtype=torch.float64, device=DEV)
        with torch.no_grad():
            for tiles, L in self.chunks():
                out, at = self.blend(self.feat, tiles, L)
                img[at] = out
        return img.view(self.H, self.W, 5)

    def backward(self, dimg):
        """Gradient of sum(dimg * image) with respect to the leaves the view was made of (accumulated in .grad)."""
        dimg = dimg.reshape(-1, 5)
        leaf = self.feat.detach()
        total = torch.zeros_like(leaf)
        for tiles, L in self.chunks():
            f = leaf.clone().requires_grad_()
            out, at = self.blend(f, tiles, L)
            total += torch.autograd.grad(out, f, dimg[at])[0]
        self.feat.backward(total)


def _blur(x):
    """11-tap Gaussian (sigma 1.5), zero padding, both ways; x: C x H x W."""
    k = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / 4.5)
    k = k / k.sum()
    for dim in (1, 2):
        n = x.shape[dim]
        pad = [5, 5, 0, 0] if dim == 2 else [0, 0, 5, 5]
        p = torch.nn.functional.pad(x, pad)
        x = sum(k[i] * p.narrow(dim, i, n) for i in range(11))
    return x


def _exact_loss(rgb, tgt, E, lam=0.2):
    x = (rgb @ E[:, :3].T + E[:, 3]).permute(2, 0, 1)
    y = tgt.permute(2, 0, 1)
    mx, my = _blur(x), _blur(y)
    sxx, syy, sxy = _blur(x * x) - mx * mx, _blur(y * y) - my * my, _blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = (2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))
    return (1 - lam) * (x - y).abs().mean() + lam * (1 - ssim.mean())


def _exact_grad_of_loss(rgb, tgt, E):
    """(loss, dL/drgb, dL/dE) in 64 bits."""
    rgb, E = rgb.detach().requires_grad_(), E.detach().requires_grad_()
    loss = _exact_loss(rgb, tgt, E)
    dC, dE = torch.autograd.grad(loss, (rgb, E))
    return loss.detach(), dC, dE


def _leaves64(params):
    return {k: v.detach().double().requires_grad_() for k, v in params.items()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        rgb, tgt, E = (t.double() for t in _loss_inputs(case, seed))
        loss, dC, dE = _exact_grad_of_loss(rgb, tgt, E)
        return dict(loss=loss.reshape(1), dC=dC, dE=dE)
    if kind == "grad":
        params, cam, img, twist, E, gD, gO = _grad_inputs(case, seed)
        p, tw, E64 = _leaves64(params), twist.double().requires_grad_(), E.double()
        view = _Exact(p, cam, case["tile"], tw)
        out = view.image()
        loss, dC, dE = _exact_grad_of_loss(out[..., :3], img.double(), E64)
        d = torch.zeros_like(out)
        d[..., :3] = dC
        if gD is not None:
            d[..., 3], d[..., 4] = gD.double(), gO.double()
        view.backward(d)
        return dict(rgb=out[..., :3], depth=out[..., 3], opacity=out[..., 4], loss=loss, grads=[p[k].grad for k in NAMES] + [tw.grad, dE])
    if kind == "render":
        params, cams, _, _, _ = _scene(case, seed, targets=False)
        with torch.no_grad():
            out = _Exact({k: v.double() for k, v in params.items()}, cams[0], 16).image()
        return dict(rgb=out[..., :3], depth=out[..., 3], opacity=out[..., 4])
    if kind == "expand":
        params, cam, xyz, rgb = _expand_inputs(case, seed)
        with torch.no_grad():
            opac = _Exact({k: v.double() for k, v in params.items()}, cam, 16).image()[..., 4]
        R, t = torch.tensor(np.asarray(cam["R"]), device=DEV), torch.tensor(np.asarray(cam["t"]), device=DEV)
        pc = xyz.double() @ R.T + t
        z = pc[:, 2]
        u, v = torch.floor(cam["fx"] * pc[:, 0] / z + cam["cx"] + 0.5), torch.floor(cam["fy"] * pc[:, 1] / z + cam["cy"] + 0.5)
        ok = (z > 0.2) & (u >= 0) & (u < cam["width"]) & (v >= 0) & (v < cam["height"])
        at = torch.where(ok, v * cam["width"] + u, torch.zeros_like(u)).long()
        keep = ok & (opac.reshape(-1)[at] < 0.99)
        m = int(keep.sum())
        new = dict(means=xyz[keep].double(), log_scales=torch.log(z[keep] / cam["fx"])[:, None].expand(m, 3),
                   quats=torch.tensor([1.0, 0, 0, 0], dtype=torch.float64, device=DEV).expand(m, 4),
                   logits=torch.full((m,), math.log(0.1 / 0.9), dtype=torch.float64, device=DEV))
        sh = torch.zeros((m,) + tuple(params["sh"].shape[1:]), dtype=torch.float64, device=DEV)
        sh[:, 0] = (rgb[keep].double() - 0.5) / (0.5 / math.sqrt(math.pi))
        new["sh"] = sh
        rest = {k: torch.zeros((case["points"] - m,) + tuple(v.shape[1:]), dtype=torch.float64, device=DEV) for k, v in params.items()}
        return dict(added=None, params={k: torch.cat([params[k].double(), new[k], rest[k]]) for k in NAMES})
    # one step from zero moments: p - lr g / (|g| + eps)
    params, cams, imgs, _, _ = _scene(case, seed)
    p = _leaves64(params)
    views = _windows(case, cams)[0]
    E0 = torch.cat([torch.eye(3, dtype=torch.float64, device=DEV), torch.zeros(3, 1, dtype=torch.float64, device=DEV)], 1)
    seen = torch.zeros(case["n"], dtype=torch.bool, device=DEV)
    loss, exposure = 0.0, []
    for k in views:
        view = _Exact(p, cams[k], 16)
        out = view.image()
        L, dC, dE = _exact_grad_of_loss(out[..., :3], imgs[k].double(), E0)
        d = torch.zeros_like(out)
        d[..., :3] = dC / len(views)
        view.backward(d)
        seen |= view.visible
        loss += float(L) / len(views)
        gE = dE / len(views)
        exposure.append(E0 - LR["exposure"] * gE / (gE.abs() + EPS))
    if not case["sparse"]:
        seen[:] = True
    new = {}
    for k in NAMES:
        g = p[k].grad
        lr = torch.full((1,), LR.get(k, 0.0), dtype=torch.float64, device=DEV)
        if k == "sh":
            lr = torch.full((g.shape[1], 1), LR["rest"], dtype=torch.float64, device=DEV)
            lr[0] = LR["dc"]
        g = torch.where(seen.view((-1,) + (1,) * (g.dim() - 1)), g, torch.zeros_like(g))
        new[k] = p[k].detach() - lr * g / (g.abs() + EPS)
    return dict(loss=loss, exposure=exposure, params=new)
