"""The training kernel's tiling: 16 samples per warp, 128 per block, and sets larger than the
grid, whose CTAs loop over blocks; gradients against the FP64 oracle at the edges of each,
and features at an address that only 4-byte loads fit."""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _data(N, seed):
    rng = np.random.default_rng(seed)
    F = (1.5 * rng.standard_normal((N, 16))).astype(np.float32)
    y = (rng.random(N) < 0.4).astype(np.float32)
    return F, y


@pytest.mark.parametrize("N", [16, 17, 127, 128, 129, 152 * 128 - 1, 152 * 128 + 1, 70001])
def test_gradient_at_tile_and_grid_edges(N):
    import paper_1704_09012_gb300 as rl0
    F, y = _data(N, N)
    w = rl0.mlp_init(seed=3)
    Fd, yd = torch.from_numpy(F).cuda(), torch.from_numpy(y).cuda()
    loss, g = rl0.mlp_grad(w, Fd, yd)
    Lo, go = omlp.loss_and_grad(w.cpu().numpy().astype(np.float64), F.astype(np.float64), y.astype(np.float64))
    # FP32 logits carry about 1e-6 of error, which the mean over samples does not raise
    assert loss == pytest.approx(Lo, rel=1e-6)
    assert np.linalg.norm(g.cpu().numpy().astype(np.float64) - go) <= 1e-5 * np.linalg.norm(go)
    # one float further on: 4-byte loads of the features, the same arithmetic
    shifted = torch.empty(16 * N + 1, device="cuda")[1:].view(N, 16)
    shifted.copy_(Fd)
    loss1, g1 = rl0.mlp_grad(w, shifted, yd)
    assert loss1 == loss and torch.equal(g1, g)


def test_training_follows_the_gradient():
    """Two Adam steps (the second of a ragged minibatch) against Adam on the oracle's gradient."""
    import paper_1704_09012_gb300 as rl0
    F, y = _data(500, 1)
    w = rl0.mlp_init(seed=5)
    w64 = w.cpu().numpy().astype(np.float64)
    rl0.mlp_train(w, torch.from_numpy(F).cuda(), torch.from_numpy(y).cuda(), epochs=1, batch=300, lr=1e-3)
    m = v = np.zeros_like(w64)
    for step, (a, b) in enumerate([(0, 300), (300, 500)], 1):
        _, g = omlp.loss_and_grad(w64, F[a:b].astype(np.float64), y[a:b].astype(np.float64))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w64 = w64 - 1e-3 * (m / (1 - 0.9 ** step)) / (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    # a step is at most lr per parameter, whatever the gradient's size: where the gradient is
    # far above its rounding, the two agree to a small part of lr
    big = np.sqrt(v) > 1e-4 * np.sqrt(v).max()
    assert np.max(np.abs(w.cpu().numpy() - w64)[big]) <= 0.02 * 1e-3
