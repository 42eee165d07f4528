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
