"""The reductions behind the loss and the pose gradient: their kernels' splits
at the smallest sizes, where the CTAs of a cluster finish as they start."""
import numpy as np
import pytest

import oracle

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
