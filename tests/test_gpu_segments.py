"""Split tiles: a tile list of at least 2 S Gaussians rendered and
back-propagated as segments of S Gaussians by separate warps, the
transmittance combined as a product of per-segment products.  With S = 64
the test scenes split many tiles; renders, contributor counts and gradients
must still equal the oracle (float32 rounding of the transmittance product
stays inside the ambiguity windows of the skip/stop decisions)."""
import numpy as np
import pytest

import oracle
from paper_2404_06926_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PIX_TOL = 1e-5
CASES = [(16, 1, 64, 0), (16, 2, 64, 1), (8, 1, 64, 0), (32, 4, 128, 1), (16, 1, 128, 1)]


def _dev(params):
    return {k: torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda() for k, v in params.items()}


def _rel(gpu, ref, floor_frac=1e-4):
    gpu = np.asarray(gpu, np.float64).ravel()
    ref = np.asarray(ref, np.float64).ravel()
    floor = floor_frac * max(np.abs(ref).max(), 1e-30)
    r = np.abs(gpu - ref) / np.maximum(np.abs(ref), floor)
    return float(np.median(r)), float(np.percentile(r, 99))


def _split_tiles(ctx, cam, tile, seg):
    TX, TY = (cam["width"] + tile - 1) // tile, (cam["height"] + tile - 1) // tile
    _, _, ranges = ctx.instances(TX * TY, "cuda")
    L = (ranges[:, 1] - ranges[:, 0]).cpu().numpy()
    return int((L >= 2 * seg).sum())


@pytest.mark.parametrize("scene", ["small_frustum", "diff_check"])
@pytest.mark.parametrize("tile,ppl,seg,persistent", CASES)
def test_split_render_parity(scene, tile, ppl, seg, persistent):
    from paper_2404_06926_gb300 import binding
    sc = getattr(scenes, scene)()
    cam = sc["cam"]
    _, _, img = oracle.forward(sc["params"], cam, tile)
    ctx = binding.Ctx()
    ctx.set_exec(segment=seg, pixels_per_lane=ppl, persistent=persistent)
    rgb, dep, opa = ctx.forward(_dev(sc["params"]), cam, tile)
    assert _split_tiles(ctx, cam, tile, seg) > 0
    T, nc = ctx.pixel_state(cam["height"], cam["width"], "cuda")
    ok = img["ambiguous"] == 0
    assert ok.mean() > 0.99
    rgb, dep, opa, T, nc = (x.cpu().numpy() for x in (rgb, dep, opa, T, nc))
    assert np.abs(rgb - img["color"])[ok].max() <= PIX_TOL
    assert np.abs(opa - img["opacity"])[ok].max() <= PIX_TOL
    assert np.abs(T - img["T_final"])[ok].max() <= PIX_TOL
    zmax = max(1.0, float(np.abs(img["depth"]).max()))
    assert np.abs(dep - img["depth"])[ok].max() <= PIX_TOL * zmax
    assert np.array_equal(nc[ok], img["n_contrib"][ok])


@pytest.mark.parametrize("scene", ["small_frustum", "diff_check"])
@pytest.mark.parametrize("extra", [False, True])
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("pg", [0, 1], ids=["per_pixel", "per_gaussian"])
def test_split_gradient_parity(scene, extra, det, pg):
    from paper_2404_06926_gb300 import binding
    sc = getattr(scenes, scene)()
    cam = sc["cam"]
    pre, bins, img = oracle.forward(sc["params"], cam, 16)
    rng = np.random.default_rng(21)
    H, W = cam["height"], cam["width"]
    dC = (rng.normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    dD = (rng.normal(size=(H, W)) * 1e-4).astype(np.float32) if extra else None
    dO = (rng.normal(size=(H, W)) * 1e-3).astype(np.float32) if extra else None
    g = oracle.backward(sc["params"], cam, pre, bins, dC.astype(np.float64),
                        None if dD is None else dD.astype(np.float64),
                        None if dO is None else dO.astype(np.float64))
    p = _dev(sc["params"])
    ctx = binding.Ctx()
    ctx.set_exec(segment=64, deterministic=det, per_gaussian=pg)
    ctx.forward(p, cam, 16)
    assert _split_tiles(ctx, cam, 16, 64) > 0
    tt = lambda a: None if a is None else torch.from_numpy(a).cuda()
    gg, pose = ctx.backward(p, tt(dC), tt(dD), tt(dO))
    vis = pre["radius"] > 0
    for name in ("means", "log_scales", "quats", "logits", "sh"):
        a = gg[name].cpu().numpy()
        assert np.all(a[~vis] == 0), name
        med, p99 = _rel(a[vis], g[name][vis])
        assert med < 1e-3 and p99 < 1e-2, (name, med, p99)
    pose = pose.cpu().numpy().astype(np.float64)
    rel = np.abs(pose - g["pose"]) / np.maximum(np.abs(g["pose"]), 1e-4 * np.abs(g["pose"]).max())
    assert np.median(rel) < 1e-3 and rel.max() < 1e-2, (pose, g["pose"], rel)


def test_split_window_step_with_graphs_matches_oracle():
    from paper_2404_06926_gb300 import binding
    sc = scenes.diff_check()
    base = sc["cam"]
    rng = np.random.default_rng(31)
    cams, targets = [], []
    for (W, H, f) in ((256, 192, 200.0), (192, 128, 150.0), (160, 160, 170.0)):
        R = scenes._rodrigues(rng.normal(0, 0.02, 3)) @ np.asarray(base["R"])
        t = np.asarray(base["t"]) + rng.normal(0, 0.05, 3)
        cams.append(scenes.camera(W, H, f, f, W / 2, H / 2, R=R, t=t))
        targets.append(rng.uniform(0, 1, (H, W, 3)).astype(np.float32))
    params = sc["params"]
    views = [(10 + i, cams[i], targets[i]) for i in range(3)]
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=3, tile_size=16, capacity_hint=8192))
    m.set_params(params)
    m.set_exec(segment=64, use_graphs=1, persistent=1)
    loss = m.optimize_step(views, want_loss=True)
    st = oracle.new_window_state(params, 3)
    r = oracle.optimize_window(params, st, cams, targets, step=1, Ts=16)
    assert abs(loss - r["loss"]) <= 2e-5 * r["loss"]
    got = m.get_params()
    vis = r["visible"]
    for name in ("means", "log_scales", "quats", "logits"):
        d_gpu = got[name].astype(np.float64) - params[name]
        d_or = st["p"][name] - params[name]
        gref = r["grads"][name][vis]
        clear = np.abs(gref) > 1e-3 * np.sqrt(np.mean(gref ** 2))
        agree = np.abs(d_gpu[vis] - d_or[vis])[clear] <= 1e-3 * oracle.DEFAULT_LR[name] + 1e-7
        assert agree.mean() > 0.99, (name, agree.mean())
    # a replayed segmented step equals an eager one (deterministic backward)
    a, b = (binding.Map(binding.default_config(n_sky=0, sh_degree=3, tile_size=16, capacity_hint=8192))
            for _ in range(2))
    for mm, graphs in ((a, 0), (b, 1)):
        mm.set_params(params)
        mm.set_exec(segment=64, use_graphs=graphs, deterministic=1)
        for _ in range(3):
            mm.optimize_step(views)
    pa, pb = a.get_params(), b.get_params()
    for k in pa:
        assert np.array_equal(pa[k], pb[k]), k


@pytest.mark.parametrize("scene", ["small_frustum", "diff_check"])
@pytest.mark.parametrize("bd", [128, 256])
def test_deep_batches_render_and_gradients(scene, bd):
    """Batches of 128 and 256 records per warp (segments of 64, so the split
    tiles' replay pass runs them too): pixels and gradients equal the oracle."""
    from paper_2404_06926_gb300 import binding
    sc = getattr(scenes, scene)()
    cam = sc["cam"]
    pre, bins, img = oracle.forward(sc["params"], cam, 16)
    H, W = cam["height"], cam["width"]
    dC = (np.random.default_rng(22).normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    g = oracle.backward(sc["params"], cam, pre, bins, dC.astype(np.float64))
    p = _dev(sc["params"])
    ctx = binding.Ctx()
    ctx.set_exec(segment=64, batch_depth=bd, persistent=1)
    rgb, _, _ = ctx.forward(p, cam, 16)
    ok = img["ambiguous"] == 0
    assert np.abs(rgb.cpu().numpy() - img["color"])[ok].max() <= PIX_TOL
    gg, _ = ctx.backward(p, torch.from_numpy(dC).cuda())
    vis = pre["radius"] > 0
    for name in ("means", "log_scales", "quats", "logits", "sh"):
        med, p99 = _rel(gg[name].cpu().numpy()[vis], g[name][vis])
        assert med < 1e-3 and p99 < 1e-2, (name, med, p99)


def test_segment_zero_keeps_lists_whole():
    """segment = 0 never splits: the images and pixel states of a deep list are
    those of a segment longer than the list, bit for bit; a context that was
    told nothing splits at 512; -1 asks for that again; other values are refused."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(3)
    n = 3000
    cam = scenes.camera(20, 13, 100.0, 100.0, 10.0, 6.5)
    params = dict(means=np.stack([rng.normal(0, 0.05, n), rng.normal(0, 0.05, n), rng.uniform(1, 3, n)], 1),
                  log_scales=rng.uniform(0.4, 0.8, (n, 3)), quats=rng.normal(size=(n, 4)),
                  logits=np.full(n, -5.0), sh=rng.normal(0, 0.5, (n, 1, 3)))
    p = {k: torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda() for k, v in params.items()}

    def images(seg):
        ctx = binding.Ctx()
        if seg is not None:
            ctx.set_exec(segment=seg)
        out = list(ctx.forward(p, cam, 16)) + list(ctx.pixel_state(13, 20, "cuda"))
        return [x.cpu().numpy() for x in out]

    same = lambda a, b: all(np.array_equal(x, y) for x, y in zip(a, b))
    whole, split = images(65536), images(512)
    assert not same(whole, split)   # the rounding of the products tells them apart
    assert same(images(0), whole)
    assert same(images(None), split) and same(images(-1), split)
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, capacity_hint=n))
    assert m.get_exec()["segment"] == -1
    assert m.set_exec(segment=0)["segment"] == 0 and m.get_exec()["segment"] == 0
    for bad in (-2, 1, 63, 96, 131072):
        with pytest.raises(binding.GLError, match="INVALID"):
            m.set_exec(segment=bad)
        with pytest.raises(binding.GLError, match="INVALID"):
            binding.Ctx().set_exec(segment=bad)


def _deep_wide(n=6000, W=320, H=240):
    """Lists of over a thousand Gaussians in the tiles of 32 pixels around the centre."""
    rng = np.random.default_rng(11)
    cam = scenes.camera(W, H, 200.0, 200.0, W / 2, H / 2)
    params = dict(means=np.stack([rng.normal(0, 0.3, n), rng.normal(0, 0.25, n), rng.uniform(2, 3, n)], 1),
                  log_scales=rng.uniform(-1.6, -1.0, (n, 3)), quats=rng.normal(size=(n, 4)),
                  logits=np.full(n, -5.0), sh=rng.normal(0, 0.5, (n, 1, 3)))
    return cam, {k: np.ascontiguousarray(v, np.float32) for k, v in params.items()}


def test_lists_stay_whole_where_the_state_finds_no_memory():
    """Where the split tiles' state is refused memory, the default execution keeps
    lists whole, without an error and without asking again for 64 calls; an
    explicit segment reports it.  Memory that comes back is used again."""
    from paper_2404_06926_gb300 import binding
    cam, params = _deep_wide()
    p = {k: torch.from_numpy(v).cuda() for k, v in params.items()}
    limit = 2 << 20   # above every other buffer (records 16 bytes an instance), below the state (96 at 32 x 32 tiles)

    def forward(ctx):
        out = list(ctx.forward(p, cam, 32)) + list(ctx.pixel_state(cam["height"], cam["width"], "cuda"))
        return [x.cpu().numpy() for x in out]

    same = lambda a, b: all(np.array_equal(x, y) for x, y in zip(a, b))
    whole, split = binding.Ctx(), binding.Ctx()
    whole.set_exec(segment=0)
    ref_whole, ref_split = forward(whole), forward(split)
    inst = whole.num_instances()
    assert 16 * 1.25 * inst + 4096 < limit < 96 * inst and not same(ref_whole, ref_split)
    dC = torch.from_numpy(np.random.default_rng(1).normal(size=(cam["height"], cam["width"], 3)).astype(np.float32)).cuda()
    ctx, told = binding.Ctx(), binding.Ctx()
    told.set_exec(segment=512)
    told.forward(p, cam, 8)   # everything but the state for 32 x 32 tiles
    m = binding.Map(binding.default_config(n_sky=0, sh_degree=0, tile_size=32, capacity_hint=len(params["logits"])))
    m.set_params(params)
    try:
        binding.selftest_alloc_limit(limit)
        for _ in range(10):
            assert same(forward(ctx), ref_whole)
        grads, _ = ctx.backward(p, dC)
        assert binding.selftest_alloc_limit(limit) == 1
        with pytest.raises(binding.GLError, match="OOM"):
            told.forward(p, cam, 32)
        binding.selftest_alloc_limit(limit)
        for graphs in (0, 1):
            m.set_exec(use_graphs=graphs)
            losses = [m.optimize_step([(1, cam, np.zeros((cam["height"], cam["width"], 3), np.float32))], want_loss=True)
                      for _ in range(4)]
            assert all(np.isfinite(losses)) and losses[3] < losses[0]
        assert binding.selftest_alloc_limit(limit) == 1
    finally:
        binding.selftest_alloc_limit(0)
    ref, _ = whole.backward(p, dC)
    for k in grads:   # the order of float atomics
        a, b = grads[k].double(), ref[k].double()
        assert float((a - b).norm() / b.norm()) < 1e-3, k
    # ten calls were made, fewer than 64 more until the state is asked for again
    for _ in range(64):
        out = forward(ctx)
    assert same(out, ref_split)
