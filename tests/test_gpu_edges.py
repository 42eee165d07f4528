"""Kernels at the sizes where their splits and tiles end: hit counts around the
backward's groups of sixteen, lists around the runs, rounds and segments of a
split tile, loss images around the 32 x 32 tile and its halo, Gaussian counts
around a warp's, copies of odd length and alignment.  Against the oracle, with
the tolerances of the parity tests (pixels 1e-5; gradients: median relative
error 1e-3, 99th percentile 1e-2, floor 1e-4 of the largest)."""
import numpy as np
import pytest

import oracle
from paper_2404_06926_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NAMES = ("means", "log_scales", "quats", "logits", "sh")


def _dev(params):
    return {k: torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda() for k, v in params.items()}


def _stack(n, opacity, seed=0):
    """n wide Gaussians behind one another, each covering the whole 20 x 13 image."""
    rng = np.random.default_rng(seed)
    cam = scenes.camera(20, 13, 100.0, 100.0, 10.0, 6.5)
    z = rng.permutation(np.linspace(1.0, 3.0, n)) if n > 1 else np.array([2.0])
    q = rng.normal(size=(n, 4))
    return cam, dict(means=np.stack([rng.normal(0, 0.05, n), rng.normal(0, 0.05, n), z], 1).astype(np.float32),
                     log_scales=rng.uniform(0.4, 0.8, (n, 3)).astype(np.float32),
                     quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                     logits=np.full(n, np.log(opacity / (1 - opacity)), np.float32),
                     sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32))


def _check_stack(n, opacity, extra, tile=16, **knobs):
    from paper_2404_06926_gb300 import binding
    cam, params = _stack(n, opacity)
    H, W = cam["height"], cam["width"]
    pre, bins, img = oracle.forward(params, cam, tile)
    rng = np.random.default_rng(n)
    dC = (rng.normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    dD = (rng.normal(size=(H, W)) * 1e-4).astype(np.float32) if extra else None
    dO = (rng.normal(size=(H, W)) * 1e-3).astype(np.float32) if extra else None
    g = oracle.backward(params, cam, pre, bins, dC.astype(np.float64), None if dD is None else dD.astype(np.float64),
                        None if dO is None else dO.astype(np.float64))
    ctx = binding.Ctx()
    ctx.set_exec(**knobs)
    p = _dev(params)
    rgb, dep, opa = ctx.forward(p, cam, tile)
    T, nc = ctx.pixel_state(H, W, "cuda")
    ok = img["ambiguous"] == 0
    assert ok.mean() > 0.9
    assert np.abs(rgb.cpu().numpy() - img["color"])[ok].max() <= 1e-5
    assert np.abs(opa.cpu().numpy() - img["opacity"])[ok].max() <= 1e-5
    assert np.abs(T.cpu().numpy() - img["T_final"])[ok].max() <= 1e-5
    assert np.abs(dep.cpu().numpy() - img["depth"])[ok].max() <= 3e-5
    assert np.array_equal(nc.cpu().numpy()[ok], img["n_contrib"][ok])
    tt = lambda a: None if a is None else torch.from_numpy(a).cuda()
    gg, _ = ctx.backward(p, tt(dC), tt(dD), tt(dO))
    for name in NAMES:
        a, ref = gg[name].cpu().numpy().astype(np.float64).ravel(), np.asarray(g[name], np.float64).ravel()
        rel = np.abs(a - ref) / np.maximum(np.abs(ref), 1e-4 * max(np.abs(ref).max(), 1e-30))
        assert np.median(rel) < 1e-3 and np.percentile(rel, 99) < 1e-2, (name, np.median(rel), np.percentile(rel, 99))


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 32, 33, 65])
@pytest.mark.parametrize("ppl,det,extra,pg", [(1, 0, False, 0), (1, 0, True, 0), (2, 0, True, 0), (4, 0, False, 0),
                                              (1, 1, True, 0), (1, 1, False, 1)])
def test_backward_hit_counts(n, ppl, det, extra, pg):
    _check_stack(n, 0.05, extra, pixels_per_lane=ppl, deterministic=det, per_gaussian=pg)


@pytest.mark.parametrize("W,H", [(1, 1), (5, 40), (31, 33), (32, 32), (33, 31), (52, 53), (84, 107)])
def test_loss_sizes(W, H):
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(W * 1000 + H)
    C = rng.uniform(0, 1, (H, W, 3)).astype(np.float32)
    tgt = np.clip(C + rng.normal(0, 0.1, (H, W, 3)), 0, 1).astype(np.float32)
    E = (np.eye(3, 4) + rng.normal(0, 0.05, (3, 4))).astype(np.float32)
    L = oracle.loss(C.astype(np.float64), tgt, E)
    ctx = binding.Ctx()
    loss, dC, dE = ctx.loss(*(torch.from_numpy(x).cuda() for x in (C, tgt, E.reshape(12))))
    assert abs(loss.item() - L["loss"]) <= 1e-5 * abs(L["loss"])
    for got, ref in ((dC, L["dL_dC"]), (dE, L["dL_dE"])):
        a, ref = got.cpu().numpy().astype(np.float64).ravel(), np.asarray(ref, np.float64).ravel()
        rel = np.abs(a - ref) / np.maximum(np.abs(ref), 1e-4 * np.abs(ref).max())
        assert np.median(rel) < 1e-3 and np.percentile(rel, 99) < 1e-2, (np.median(rel), np.percentile(rel, 99))


@pytest.mark.parametrize("n", [127, 128, 129, 192, 511, 512, 513, 577, 1030, 1100])
@pytest.mark.parametrize("opacity", [0.006, 0.4])   # no pixel stops (0.994^1100 > 1e-4); every pixel stops early
@pytest.mark.parametrize("ppl,persistent", [(1, 0), (2, 1)])
def test_split_list_lengths(n, opacity, ppl, persistent):
    _check_stack(n, opacity, True, segment=64, pixels_per_lane=ppl, persistent=persistent)


@pytest.mark.parametrize("seg", [64, 256, 1024])
@pytest.mark.parametrize("bd", [32, 64, 256])
def test_split_segments_of_several_runs(seg, bd):
    _check_stack(2100, 0.02, False, segment=seg, batch_depth=bd)


@pytest.mark.parametrize("n", [1, 3, 683, 2731, 5000])   # around the copy's chunk of 8192 floats
def test_parameter_copies(n):
    """Parameters set and read back (aligned, and rows into the middle of larger
    arrays), and a new map's moments, are exact."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    p = _dev(dict(means=rng.normal(size=(n, 3)), log_scales=rng.normal(size=(n, 3)), quats=rng.normal(size=(n, 4)),
                  logits=rng.normal(size=n), sh=rng.normal(size=(n, 4, 3))))
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=1, capacity_hint=n))
    m.set_params(p)
    out = m.get_params()
    host = {k: np.zeros(v.shape, np.float32) for k, v in p.items()}
    gs = binding.gaussians(host)
    binding.check(binding.lib().gl_map_get_params(m._h, binding.C.byref(gs), None))
    odd = {k: torch.zeros(v.numel() + 1, device="cuda") for k, v in p.items()}
    go = binding.gaussians({k: v[1:].view(p[k].shape) for k, v in odd.items()})   # 4-byte aligned only
    binding.check(binding.lib().gl_map_get_params(m._h, binding.C.byref(go), None))
    torch.cuda.synchronize()
    for k in NAMES:
        assert torch.equal(torch.as_tensor(out[k]).cpu().reshape(-1), p[k].cpu().reshape(-1)), k
        assert np.array_equal(host[k], p[k].cpu().numpy()), k
        assert torch.equal(odd[k][1:], p[k].reshape(-1)) and odd[k][0] == 0, k
    for which in (1, 2):
        assert all(float(torch.as_tensor(v).abs().max()) == 0 for v in m.get_moments(which).values())


def test_render_into_device_images():
    """Images rendered in place equal those copied to the host, also where two
    of them share memory (the later copy wins)."""
    from paper_2404_06926_gb300 import binding
    sc = scenes.small_frustum(n=300)
    cam = sc["cam"]
    H, W = cam["height"], cam["width"]
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=300))
    m.set_params(_dev(sc["params"]))
    hd, ho = np.empty((H, W), np.float32), np.empty((H, W), np.float32)
    hc = m.render(cam, out_depth=hd, out_opacity=ho)
    c, d, o = (torch.empty(s, device="cuda") for s in ((H, W, 3), (H, W), (H, W)))
    m.render(cam, out_rgb=c, out_depth=d, out_opacity=o)
    assert np.array_equal(c.cpu().numpy(), hc) and np.array_equal(d.cpu().numpy(), hd)
    assert np.array_equal(o.cpu().numpy(), ho)
    m.render(cam, out_rgb=c, out_depth=d, out_opacity=d)
    assert np.array_equal(d.cpu().numpy(), ho)
    E = np.concatenate([np.eye(3, dtype=np.float32), np.full((3, 1), 0.25, np.float32)], 1)
    m.render(cam, E=E, out_rgb=c)
    assert np.allclose(c.cpu().numpy(), hc + 0.25, atol=1e-6)


@pytest.mark.parametrize("n", [1023, 1024, 1500])
def test_default_execution_splits_deep_lists(n):
    _check_stack(n, 0.02, True)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 257])
@pytest.mark.parametrize("tile", [8, 16])
def test_exact_culling_of_mixed_rectangles(n, tile):
    """Rectangles from one tile to more than 64 within a warp: the instances
    are the oracle's, bit for bit."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    cam = scenes.camera(203, 151, 150.0, 150.0, 101.0, 75.0)
    z = rng.uniform(0.1, 6.0, n)   # some behind the near plane
    q = rng.normal(size=(n, 4))
    params = dict(means=np.stack([rng.uniform(-0.8, 0.8, n) * z, rng.uniform(-0.6, 0.6, n) * z, z], 1).astype(np.float32),
                  log_scales=rng.uniform(-5.0, -0.5, (n, 3)).astype(np.float32),
                  quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                  logits=rng.normal(0, 2, n).astype(np.float32), sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32))
    pre, bins, _ = oracle.forward(params, cam, tile)
    ctx = binding.Ctx()
    ctx.forward(_dev(params), cam, tile)
    TX, TY = -(-cam["width"] // tile), -(-cam["height"] // tile)
    out = ctx.preprocess(n, "cuda")
    vis = pre["radius"] > 0
    assert np.array_equal(out["radius"].cpu().numpy(), pre["radius"])
    assert np.array_equal(out["rect"].cpu().numpy()[vis], pre["rect"][vis])
    assert not out["rect"].cpu().numpy()[~vis].any()
    assert ctx.num_instances() == bins["I"]
    keys, vals, _ = ctx.instances(TX * TY, "cuda")
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), bins["keys"])
    assert np.array_equal(vals.cpu().numpy().view(np.uint32), bins["vals"])


@pytest.mark.parametrize("n,seg", [(60, 0), (700, 0), (700, 64)])
@pytest.mark.parametrize("extra", [False, True])
def test_backward_with_more_blocks_than_warps(n, seg, extra):
    """A frame large enough for the half-warp backward (3,192 pixel blocks), of
    ragged size, with Gaussians from under a pixel to half the frame."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    W, H = 331, 300
    cam = scenes.camera(W, H, 250.0, 250.0, W / 2, H / 2)
    z = rng.uniform(1.0, 6.0, n)
    q = rng.normal(size=(n, 4))
    params = dict(means=np.stack([rng.uniform(-0.7, 0.7, n) * z, rng.uniform(-0.6, 0.6, n) * z, z], 1).astype(np.float32),
                  log_scales=rng.uniform(-6.0, -0.5, (n, 3)).astype(np.float32),
                  quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                  logits=rng.normal(0, 1.5, n).astype(np.float32), sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32))
    pre, bins, img = oracle.forward(params, cam, 16)
    dC = (rng.normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    dD = (rng.normal(size=(H, W)) * 1e-4).astype(np.float32) if extra else None
    dO = (rng.normal(size=(H, W)) * 1e-3).astype(np.float32) if extra else None
    g = oracle.backward(params, cam, pre, bins, dC.astype(np.float64), None if dD is None else dD.astype(np.float64),
                        None if dO is None else dO.astype(np.float64))
    ctx = binding.Ctx()
    ctx.set_exec(segment=seg, persistent=1 if seg else 0)
    p = _dev(params)
    ctx.forward(p, cam, 16)
    tt = lambda a: None if a is None else torch.from_numpy(a).cuda()
    gg, _ = ctx.backward(p, tt(dC), tt(dD), tt(dO))
    vis = pre["radius"] > 0
    for name in NAMES:
        a, ref = gg[name].cpu().numpy().astype(np.float64)[vis].ravel(), np.asarray(g[name], np.float64)[vis].ravel()
        rel = np.abs(a - ref) / np.maximum(np.abs(ref), 1e-4 * np.abs(ref).max())
        assert np.median(rel) < 1e-3 and np.percentile(rel, 99) < 1e-2, (name, np.median(rel), np.percentile(rel, 99))


@pytest.mark.parametrize("n", [2047, 2048, 2049, 6145, 799_999, 800_001])   # a tile's keys; the smaller tiles' last count
def test_sort_tile_sizes(n):
    """Binning of n Gaussians of one tile each: instances in (tile, depth, index) order."""
    from paper_2404_06926_gb300 import binding
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    cam = scenes.camera(640, 480, 500.0, 500.0, 320.0, 240.0)
    z = torch.rand(n, generator=g, device="cuda") * 2 + 1
    uv = torch.rand(n, 2, generator=g, device="cuda")
    means = torch.stack([(uv[:, 0] * 600 + 20 - 320) / 500 * z, (uv[:, 1] * 440 + 20 - 240) / 500 * z, z], 1).contiguous()
    q = torch.zeros(n, 4, device="cuda")
    q[:, 0] = 1
    p = dict(means=means, log_scales=torch.full((n, 3), -9.0, device="cuda"), quats=q,
             logits=torch.full((n,), 2.0, device="cuda"), sh=torch.zeros(n, 1, 3, device="cuda"))
    ctx = binding.Ctx()
    ctx.forward(p, cam, 16)
    keys, vals, ranges = ctx.instances(40 * 30, "cuda")
    assert len(keys) >= n
    same = keys[1:] == keys[:-1]
    assert bool((keys[1:] >= keys[:-1]).all()) and bool((vals[1:][same] > vals[:-1][same]).all())
    assert int(torch.unique(vals).numel()) == n
    assert torch.equal(ranges[:, 1] - ranges[:, 0], torch.bincount(keys >> 32, minlength=1200).int())


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1000])
@pytest.mark.parametrize("deg", [0, 3])
def test_expanded_rows(n, deg):
    """Points in front of the camera become rows in order, the others none."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    cam = scenes.camera(64, 48, 50.0, 50.0, 32.0, 24.0)
    xyz = rng.normal(0, 2, (n, 3)).astype(np.float32)
    rgb = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=deg, capacity_hint=16))
    added = m.add_points(torch.from_numpy(xyz).cuda(), torch.from_numpy(rgb).cuda(), cam, use_mask=False)
    keep = xyz[:, 2] > np.float32(0.2)
    assert added == keep.sum() == len(m)
    if added == 0:
        return
    out = {k: torch.as_tensor(v).cpu().numpy() for k, v in m.get_params().items()}
    assert np.array_equal(out["means"], xyz[keep])
    assert np.allclose(out["log_scales"], np.log(xyz[keep, 2:] / 50.0), atol=1e-6)
    assert np.allclose(out["sh"][:, 0], (rgb[keep] - 0.5) / 0.28209479177387814, atol=1e-6)
    assert not out["sh"][:, 1:].any()
    assert np.array_equal(out["quats"], np.tile(np.float32([1, 0, 0, 0]), (added, 1)))


@pytest.mark.parametrize("exposed", [False, True])
@pytest.mark.parametrize("second", ["out_depth", "out_opacity"])
def test_render_into_images_that_share_memory(exposed, second):
    """Colour, depth, opacity are written in that order, whatever the exposure:
    where two device images share memory the later one stays, as on the host."""
    from paper_2404_06926_gb300 import binding
    sc = scenes.small_frustum(n=300)
    cam = sc["cam"]
    H, W = cam["height"], cam["width"]
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=300))
    m.set_params(_dev(sc["params"]))
    E = np.concatenate([np.eye(3, dtype=np.float32), np.full((3, 1), 0.25, np.float32)], 1) if exposed else None
    for at in (0, 2):   # the colour's first and last third
        want = np.empty((3, H, W), np.float32)
        m.render(cam, E=E, out_rgb=want.reshape(H, W, 3), **{second: want[at]})
        got = torch.empty((3, H, W), device="cuda")
        m.render(cam, E=E, out_rgb=got.view(H, W, 3), **{second: got[at]})
        assert np.array_equal(got.cpu().numpy(), want), at


@pytest.mark.parametrize("n", [1, 3000, 100_000])
def test_arrays_read_back_into_shared_memory(n):
    """Parameters read back into device arrays that share memory: the arrays are
    written in their order, the later one winning, as into host memory."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    p = dict(means=rng.normal(size=(n, 3)), log_scales=rng.normal(size=(n, 3)), quats=rng.normal(size=(n, 4)),
             logits=rng.normal(size=n), sh=rng.normal(size=(n, 1, 3)))
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=n))
    m.set_params(_dev(p))

    def read(buf):
        out = dict(means=buf[:3 * n].reshape(n, 3), log_scales=buf[:3 * n].reshape(n, 3),
                   quats=buf[2 * n:6 * n].reshape(n, 4), logits=buf[5 * n:6 * n], sh=buf[n:4 * n].reshape(n, 1, 3))
        g = binding.gaussians(out, n)
        binding.check(binding.lib().gl_map_get_params(m._h, binding.C.byref(g), None))
        return buf

    want = read(np.zeros(6 * n, np.float32))
    for _ in range(5):
        assert np.array_equal(read(torch.zeros(6 * n, device="cuda")).cpu().numpy(), want)


class _Raw:
    """A device allocation of its own, of exactly so many bytes."""

    def __init__(self, nbytes):
        import ctypes
        torch.cuda.current_stream().synchronize()   # the primary context exists and is current
        self.cu, self.p = ctypes.CDLL("libcuda.so.1"), ctypes.c_uint64()
        assert self.cu.cuMemAlloc_v2(ctypes.byref(self.p), ctypes.c_size_t(nbytes)) == 0

    def free(self):
        self.cu.cuMemFree_v2(self.p)


def test_device_arrays_that_end_early_are_refused():
    """Arrays that end with their allocation are taken; one that ends 4 MB before
    its last row is refused on the host, read or written, as a copy would."""
    from paper_2404_06926_gb300 import binding
    n = 1_000_000
    rng = np.random.default_rng(5)
    rows = dict(means=3, log_scales=3, quats=4, logits=1, sh=3)
    p = {k: rng.normal(size=n * w).astype(np.float32) for k, w in rows.items()}
    host = dict(means=p["means"].reshape(n, 3), log_scales=p["log_scales"].reshape(n, 3), quats=p["quats"].reshape(n, 4),
                logits=p["logits"], sh=p["sh"].reshape(n, 1, 3))
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=n))
    m.set_params(host)
    L, C = binding.lib(), binding.C
    full = {k: _Raw(4 * n * w) for k, w in rows.items()}
    short = {k: _Raw(4 * n * w - (4 << 20) + 64) for k, w in rows.items() if 4 * n * w > (4 << 20)}

    def struct(**other):
        g = binding.gaussians(host)
        for k in rows:
            setattr(g, k, other.get(k, full[k]).p.value)
        return g

    for call in (lambda g: L.gl_map_get_params(m._h, C.byref(g), None), lambda g: L.gl_map_set_params(m._h, C.byref(g))):
        binding.check(call(struct()))
        for k, r in short.items():
            with pytest.raises(binding.GLError, match="INVALID"):
                binding.check(call(struct(**{k: r})))
        assert len(m) == n
    got = m.get_params()   # written to the raw arrays and read back from them
    assert all(np.array_equal(got[k].ravel(), p[k]) for k in rows)
    H, W = 1536, 2048
    cam = scenes.camera(W, H, 1000.0, 1000.0, 1024.0, 768.0)
    c, d = torch.empty((H, W, 3), device="cuda"), _Raw(4 * H * W)
    less = _Raw(4 * H * W - (4 << 20) + 64)
    K, P = binding.intrinsics(cam), binding.pose(cam)
    small = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=300))
    small.set_params(_dev(scenes.small_frustum(n=300)["params"]))
    render = lambda depth: binding.check(L.gl_render(small._h, C.byref(P), C.byref(K), None, c.data_ptr(), depth.p.value, None))
    render(d)
    with pytest.raises(binding.GLError, match="INVALID"):
        render(less)
    for r in (*full.values(), *short.values(), d, less):
        r.free()


def test_exposure_into_device_memory_does_not_crash():
    """An exposure is asked for in host memory; a device pointer is the driver's
    to take or refuse, not the host's to write to."""
    from paper_2404_06926_gb300 import binding
    cam = scenes.camera(32, 16, 30.0, 30.0, 16.0, 8.0)
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=16))
    m.add_keyframe(3, cam, np.zeros((16, 32, 3), np.float32))
    E = torch.full((12,), -1.0, device="cuda")
    st = binding.lib().gl_map_get_exposure(m._h, 3, E.data_ptr())
    assert np.array_equal(m.exposure(3), np.eye(3, 4, dtype=np.float32))
    if st == 0:
        assert np.array_equal(E.cpu().numpy().reshape(3, 4), np.eye(3, 4, dtype=np.float32))


@pytest.mark.parametrize("bd", [32, 64, 128, 256])
def test_batch_depth_reaches_the_backward_of_large_frames(bd):
    """Frames of more pixel blocks than resident warps (3,192): batches of 32
    records walk half-warp blocks, deeper ones the kernel that stages them."""
    from torch.profiler import ProfilerActivity, profile
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(60)
    W, H, n = 331, 300, 60
    cam = scenes.camera(W, H, 250.0, 250.0, W / 2, H / 2)
    z = rng.uniform(1.0, 6.0, n)
    q = rng.normal(size=(n, 4))
    params = dict(means=np.stack([rng.uniform(-0.6, 0.6, n) * z, rng.uniform(-0.5, 0.5, n) * z, z], 1).astype(np.float32),
                  log_scales=rng.uniform(-4.0, -2.0, (n, 3)).astype(np.float32),
                  quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                  logits=rng.normal(0, 1, n).astype(np.float32), sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32))
    pre, bins, _ = oracle.forward(params, cam, 16)
    dC = (rng.normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    g = oracle.backward(params, cam, pre, bins, dC.astype(np.float64))
    ctx = binding.Ctx()
    ctx.set_exec(batch_depth=bd)
    p, d = _dev(params), torch.from_numpy(dC).cuda()
    ctx.forward(p, cam, 16)
    names = set()
    for _ in range(4):   # (a profiler's first window can come back empty)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            gg, _ = ctx.backward(p, d)
            torch.cuda.synchronize()
        names |= {e.name for e in prof.events() if "k_raster_bwd" in e.name}
        if names:
            break
    assert len(names) == 1 and ("k_raster_bwd_half" in names.pop()) == (bd == 32)
    vis = pre["radius"] > 0
    for name in NAMES:
        a, ref = gg[name].cpu().numpy().astype(np.float64)[vis].ravel(), np.asarray(g[name], np.float64)[vis].ravel()
        rel = np.abs(a - ref) / np.maximum(np.abs(ref), 1e-4 * np.abs(ref).max())
        assert np.median(rel) < 1e-3 and np.percentile(rel, 99) < 1e-2, (name, np.median(rel), np.percentile(rel, 99))


@pytest.mark.parametrize("W,H", [(1151, 575), (1120, 608), (1151, 607)])   # 648, 665 and 684 tiles
def test_loss_around_the_line_between_its_kernels(W, H):
    """A cluster per tile below 4.5 tiles per SM (684 on 152 SMs), one CTA from there on."""
    test_loss_sizes(W, H)


@pytest.mark.parametrize("scale,small", [(-4.5, True), (-3.2, True), (-1.5, False)])
@pytest.mark.parametrize("seg,persistent", [(0, 0), (64, 1)])
@pytest.mark.parametrize("extra", [False, True])
def test_blocks_by_footprint(scale, small, seg, persistent, extra):
    """Frames of more pixel blocks than resident warps: Gaussians of up to 32
    instances each take half-warp blocks, larger ones whole-warp blocks.  Either
    way the gradients are those of the kernel that has whole-warp blocks only
    (batches of 64): the terms are the same, the sums' order is not (2-norm 1e-4)."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(7)
    W, H, n = 331, 300, 900
    cam = scenes.camera(W, H, 250.0, 250.0, W / 2, H / 2)
    z = rng.uniform(1.0, 6.0, n)
    q = rng.normal(size=(n, 4))
    params = dict(means=np.stack([rng.uniform(-0.6, 0.6, n) * z, rng.uniform(-0.5, 0.5, n) * z, z], 1).astype(np.float32),
                  log_scales=rng.uniform(scale - 0.3, scale + 0.3, (n, 3)).astype(np.float32),
                  quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                  logits=rng.normal(0, 1, n).astype(np.float32), sh=rng.normal(0, 0.5, (n, 1, 3)).astype(np.float32))
    p = _dev(params)
    t = lambda *s: torch.from_numpy(rng.normal(size=s).astype(np.float32)).cuda() * 1e-3
    d = [t(H, W, 3), t(H, W) if extra else None, t(H, W) if extra else None]
    res = []
    for bd in (32, 64):
        ctx = binding.Ctx()
        ctx.set_exec(batch_depth=bd, segment=seg, persistent=persistent)
        ctx.forward(p, cam, 16)
        visible = int((ctx.preprocess(n, "cuda")["radius"] > 0).sum())
        assert (ctx.num_instances() <= 32 * visible) == small
        res.append(ctx.backward(p, *d)[0])
    for k in NAMES:
        a, b = res[0][k].double(), res[1][k].double()
        assert float((a - b).norm()) <= 1e-4 * float(b.norm()), k
