"""The reductions behind the loss and the pose gradient: their kernels' splits
at the smallest sizes, where the CTAs of a cluster finish as they start."""
import numpy as np
import pytest

import oracle
from paper_2404_06926_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (32, 32), (33, 1), (96, 64)])
def test_loss_of_few_tiles_repeats_bit_for_bit(W, H):
    """Every CTA's sums reach the loss: it equals the oracle's, and 200 calls agree."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(W + H)
    C = rng.uniform(0, 1, (H, W, 3)).astype(np.float32)
    tgt = np.clip(C + rng.normal(0, 0.1, (H, W, 3)), 0, 1).astype(np.float32)
    E = (np.eye(3, 4) + rng.normal(0, 0.05, (3, 4))).astype(np.float32)
    ref = oracle.loss(C.astype(np.float64), tgt, E)["loss"]
    ctx = binding.Ctx()
    c, t, e = (torch.from_numpy(x).cuda() for x in (C, tgt, E.reshape(12)))
    out = torch.stack([ctx.loss(c, t, e)[0] for _ in range(200)]).cpu().numpy()
    assert (out == out[0]).all()
    assert abs(out[0] - ref) <= 1e-5 * abs(ref)


@pytest.mark.parametrize("n", [1, 33, 5_000, 5_440, 5_441, 50_000])   # 170 blocks of 32: one CTA's share
def test_pose_sum_repeats_bit_for_bit(n):
    """Every CTA's sums reach the pose gradient: with a deterministic backward 50
    calls agree, and the translation part (camera axes along the world's, zero
    twist) is the sum of the means' gradients."""
    from paper_2404_06926_gb300 import binding
    rng = np.random.default_rng(n)
    W, H = 64, 48
    cam = scenes.camera(W, H, 50.0, 50.0, 32.0, 24.0)
    z = rng.uniform(1.0, 6.0, n)
    q = rng.normal(size=(n, 4))
    params = dict(means=np.stack([rng.uniform(-0.6, 0.6, n) * z, rng.uniform(-0.45, 0.45, n) * z, z], 1).astype(np.float32),
                  log_scales=rng.uniform(-3.5, -2.5, (n, 3)).astype(np.float32),
                  quats=(q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                  logits=rng.normal(-2, 1, n).astype(np.float32), sh=rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32))
    dC = (rng.normal(size=(H, W, 3)) * 1e-3).astype(np.float32)
    p = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in params.items()}
    d = torch.from_numpy(dC).cuda()
    ctx = binding.Ctx()
    ctx.set_exec(deterministic=1)
    ctx.forward(p, cam, 16)
    res = [ctx.backward(p, d) for _ in range(50)]
    out = torch.stack([r[1] for r in res]).cpu().numpy().astype(np.float64)
    assert (out == out[0]).all() and np.abs(out[0]).max() > 0
    gm = res[0][0]["means"].cpu().numpy().astype(np.float64)
    # a Gaussian's part is rounded a few times on its way, a block's 32 are added in floats: under 16 roundings
    assert (np.abs(out[0, :3] - gm.sum(0)) <= 16 * 2.0 ** -24 * np.abs(gm).sum(0)).all(), (out[0, :3], gm.sum(0))


def test_exposure_gradient_keeps_what_cancels():
    """Partials of magnitudes 2^25, 2^15 (24 random bits) and 2^-25 in one column of
    sums, the large ones cancelling: a double sum is exact (50 bits), so the
    exposure gradient is the small ones'."""
    from paper_2404_06926_gb300 import binding
    TX, TY = 73, 3   # 73 columns of tiles share out the partials; down a column the magnitudes fall
    big = np.float32(2.0 ** 25)
    mid = np.float32(2.0 ** 15 * (1 + 0x2AB5E3 / 2.0 ** 23))
    small = np.float32(2.0 ** -25)
    sign = np.array([1.0 if c < 36 else -1.0 for c in range(72)] + [0.0], np.float32)
    val = np.stack([np.where(sign == 0, small, big), np.where(sign == 0, small, mid), np.full(TX, small)]).astype(np.float32)
    up = np.stack([np.where(sign == 0, 1, sign), np.where(sign == 0, 1, sign), np.ones(TX)])   # sign of colour - target
    tile = lambda a: np.repeat(np.repeat(a.astype(np.float32), 32, 0), 32, 1)
    C = np.repeat(tile(val)[..., None], 3, 2)
    tgt = C * (1 - 0.25 * tile(up))[..., None]
    ctx = binding.Ctx()
    E = torch.eye(3, 4, device="cuda").reshape(12).contiguous()
    _, _, dE = ctx.loss(*(torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda() for x in (C, tgt)), E, lam=0.0)
    H, W = C.shape[:2]
    g = 1.0 / (3.0 * W * H)     # lambda = 0: the gradient of mean |E[C] - target| is +-1 / N
    left = 73 + 2               # small tiles of one sign; the offsets' tiles: as many
    want = np.array([[g * 1024 * left * float(small)] * 3 + [g * 1024 * left]] * 3)
    assert np.allclose(dE.cpu().numpy(), want, rtol=1e-5, atol=0), (dE.cpu().numpy(), want)


def test_pose_sum_past_the_range_of_a_float():
    """The backward is linear in the image gradient: 2^k times the gradient gives
    2^k times the pose gradient, also where its partials' sums on the way (32 of 2.5e37
    to 5e37 of either sign) leave the range of a float and the total does not."""
    from paper_2404_06926_gb300 import binding
    f, z, n = 256.0, 2.0, 64 * 32
    cam = scenes.camera(256, 256, f, f, 128.0, 128.0)
    u, v = np.meshgrid(np.arange(8) * 32 + 16.0, np.arange(8) * 32 + 16.0)
    means = np.tile(np.float32([0, 0, -5]), (n, 1))   # one Gaussian of each block of 32 is seen
    means[::32] = np.stack([(u.ravel() - 128) * z / f, (v.ravel() - 128) * z / f, np.full(64, z)], 1)
    params = dict(means=means, log_scales=np.full((n, 3), np.log(3.0 * z / f), np.float32),
                  quats=np.tile(np.float32([1, 0, 0, 0]), (n, 1)), logits=np.zeros(n, np.float32),
                  sh=np.ones((n, 1, 3), np.float32))
    x = np.arange(256, dtype=np.float32)
    ramp = (x % 32 - 16) / 16
    parity = np.where((x // 32).astype(int) % 2 == 0, 1, -1)    # of the column: of the block's index
    dC = np.repeat(np.tile((ramp * parity)[None, :, None], (256, 1, 1)), 3, 2).astype(np.float32)
    p = {k: torch.from_numpy(np.ascontiguousarray(a)).cuda() for k, a in params.items()}

    def pose(params, d):
        ctx = binding.Ctx()
        ctx.set_exec(deterministic=1)
        ctx.forward(params, cam, 16)
        return ctx.backward(params, torch.from_numpy(np.ascontiguousarray(d)).cuda())[1].cpu().numpy().astype(np.float64)

    one = pose({k: a[:32].contiguous() for k, a in p.items()}, dC)[0]
    scale = 2.0 ** np.floor(np.log2(5e37 / abs(one)))
    want = pose(p, dC) * scale
    assert abs(one) * scale * 32 > 2 * 3.4e38 > 4 * abs(want[0])   # the case is what it says
    got = pose(p, dC * np.float32(scale))
    fits = np.abs(want) < 3e38
    assert fits[0] and np.allclose(got[fits], want[fits], rtol=1e-6, atol=1e-6 * abs(one) * scale), (got, want)
