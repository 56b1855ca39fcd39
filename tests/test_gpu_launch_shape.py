"""The FP32 fused step's launch shape: the reported tile is what a cell may hold
without the chunked path, and a cell above it collides as one below it does."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ppc", [100, 200])
def test_tile_holds_an_ordinary_cell(ppc):
    """Every shape that a box handle times stages the particles per cell and
    a margin above them (a quarter and 32, rounded to 16), less 32 at most."""
    from paper_2501_10965_gb300 import dsmc
    g = dsmc.Dsmc(W.homogeneous_box(ncells=200, ppc=ppc, dt=2e-3, precision="fp32"))
    g.dsmc_step(40)
    w, t = g.launch_shape()
    t0 = (5 * ppc // 4 + 32 + 15) // 16 * 16
    assert w in (2, 4) and t0 - 32 <= t <= t0 + 64


@pytest.mark.parametrize("calls", [(15,) * 4, (60,)])  # a warp per cell; the timed shapes
def test_collisions_above_the_tile(calls):
    """400 particles a cell of the same weight, staged whole (ppc 512) and in
    chunks with hashed collision owners (ppc 64): as many collisions, elastic and
    not, up to five standard errors of a Poisson count, and the same rotational
    energy after the relaxation up to five of a mean over the particles."""
    from paper_2501_10965_gb300 import dsmc
    nc, n = 32, 400
    runs = []
    for ppc, rho, seed in ((512, 8.0, 1), (64, 1.0, 2)):
        g = dsmc.Dsmc(W.homogeneous_box(ncells=nc, ppc=ppc, init_rho=rho, kn=0.1, dt=2e-3, precision="fp32", seed=seed,
                                        capacity=80000))
        rng = np.random.default_rng(seed)
        m = nc * n
        p = {"x": (np.repeat(np.arange(nc), n) + rng.random(m)) / nc, "y": np.zeros(m), "ir": rng.exponential(0.3, m)}
        p.update({k: rng.standard_normal(m) for k in ("vx", "vy", "vz")})
        g.set_particles({k: torch.tensor(v) for k, v in p.items()})
        for k in calls:
            g.dsmc_step(k)
        s = g.stats()
        runs.append((s["n_coll"], s["n_inel"], g.get_particles()["ir"].cpu().numpy()))
        assert len(runs[-1][2]) == m
    (c0, i0, r0), (c1, i1, r1) = runs
    assert c0 > 50000 and i0 > 5000 and r0.mean() > 0.35
    assert abs(c0 - c1) <= 5 * np.sqrt(c0 + c1) and abs(i0 - i1) <= 5 * np.sqrt(i0 + i1)
    assert abs(r0.mean() - r1.mean()) <= 5 * np.sqrt(r0.var() / r0.size + r1.var() / r1.size)
