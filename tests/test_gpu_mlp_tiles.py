"""Training kernel at the edges of its 32-sample tiles: one sample, a tile less
and more by one, and more tiles than CTAs (each CTA then sums several)."""
import numpy as np
import pytest

from oracle import mlp
from paper_1404_3363_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4096, 32 * 1024 + 33])
def test_gradient_at_tile_edges(n):
    from paper_1404_3363_gb300 import build, ivv
    build.build()
    vol = ivv.volume_for(scenes.twisted_cube(width=8, height=8))
    rng = np.random.default_rng(n)
    theta = (mlp.init(3) + 0.05 * rng.normal(size=mlp.N_PARAMS)).astype(np.float32)
    vol.set_guess_weights(0, theta)
    x, p = np.zeros((n, 4), np.float32), np.zeros((n, 4), np.float32)
    x[:, :3], p[:, :3] = rng.uniform(-1, 1, (n, 3)), rng.uniform(0, 1, (n, 3))
    loss, grad = vol.guess_loss_grad(0, torch.from_numpy(x).cuda(), torch.from_numpy(p).cuda())
    L, g = mlp.loss_grad(theta.astype(np.float64), x[:, :3].astype(np.float64), p[:, :3].astype(np.float64))
    # sums of up to 64 terms per layer and of n samples in FP32: a few 1e-6 of
    # the largest entry
    assert loss == pytest.approx(L, rel=1e-5)
    assert np.abs(grad - g).max() <= 1e-5 * np.abs(g).max()
