"""Gradient kernel of the HoT network at the edges of its tiles of 32 cells
and of its grid (152 CTAs), against the FP64 oracle with the same bfloat16
weights, and the Adam step joined to the reduction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as om
from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _data(nx, seed=0):
    from paper_2501_10965_gb300 import dsmc
    cfg = W.couette_1d(kn=0.1, nx=nx, ppc=1, kn_ref=0.0)
    g = dsmc.Dsmc(cfg)
    rng = np.random.default_rng(seed)
    x = (np.arange(nx) + 0.5) / nx
    f = np.zeros((nx, 18))
    f[:, 0] = 1.0 + 0.02 * np.sin(3 * x)
    f[:, 2] = 0.3 * (2 * x - 1) + 0.01 * np.cos(5 * x)
    f[:, 4] = 1.0 + 0.05 * x * (1 - x)
    f[:, 5] = 1.0 + 0.03 * x * (1 - x)
    hot = 0.05 * rng.standard_normal((nx, 12))
    ft = torch.tensor(f, device="cuda")
    _, kn, _ = g.dsmc_hot(ft)
    mask = torch.tensor((rng.uniform(size=nx) < 0.8).astype(np.uint8), device="cuda")
    mask[0] = 1
    theta = om.init_params(seed + 1).astype(np.float32)
    theta += (0.02 * rng.standard_normal(theta.size)).astype(np.float32)
    g.mlp_set_params(theta)
    X, sc = om.features(f, kn.cpu().numpy(), cfg)
    Y = om.targets(hot, sc)
    m = mask.cpu().numpy().astype(bool)
    th = om.bf16_round(theta)  # weights and biases in bfloat16
    loss, grad = om.loss_and_grad(th, X[m], Y[m])
    return g, (ft, torch.tensor(hot, device="cuda"), kn, mask), theta, loss, grad


@pytest.mark.parametrize("nx", [1, 31, 32, 33, 152 * 32, 152 * 32 + 1, 10000])
def test_gradient_at_tile_edges(nx):
    g, data, _, loss, grad = _data(nx)
    lg, gg = g.mlp_grad(*data)
    # FP32 sums of products over at most 64 terms and nx cells
    assert abs(lg - loss) <= 1e-5 * max(loss, 1e-6)
    assert np.linalg.norm(gg - grad) <= 1e-5 * np.linalg.norm(grad)


def test_train_step_is_adam_on_that_gradient():
    g, data, theta, _, _ = _data(1000)
    _, g0 = g.mlp_grad(*data)
    assert np.array_equal(g.mlp_get_params(), theta)
    g.mlp_train(*data, nsteps=1, lr=1e-3)
    # first Adam step: lr g / (|g| + eps), up to FP32 rounding of the moments
    want = theta - 1e-3 * g0 / (np.abs(g0) + 1e-8)
    assert np.allclose(g.mlp_get_params(), want, rtol=0, atol=2e-6)
