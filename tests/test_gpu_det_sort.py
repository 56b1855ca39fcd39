"""FP64-deterministic layout: the sort by cell (counts, scan over the grid,
lists of source slots, gather) at the sizes where its parts change: one warp
or eight per CTA, cells above the shared-memory tile, scans and lists beyond
one CTA, few or many candidates per cell."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("x", "y", "vx", "vy", "vz", "ir")


def _np(p):
    return {k: v.cpu().numpy() for k, v in p.items()}


@pytest.mark.parametrize("cfg", [
    W.fourier_1d(nx=3, ppc=300, kn=0.05),                                     # cells above the tile, one warp per CTA
    W.cavity_2d(nx=61, ny=5, ppc=9, kn=0.05, precision="fp64"),               # 305 cells: eight warps, a ragged last CTA
    W.cavity_2d(nx=18, ny=18, ppc=290, kn=0.02, precision="fp64", lx=0.2, ly=0.2, dt=1e-3),  # above the tile, eight warps
    W.cavity_2d(nx=70, ny=59, ppc=4, kn=0.05, precision="fp64"),              # 4 130 cells, 16 520 particles
    W.cavity_2d(nx=20, ny=17, ppc=60, kn=0.002, precision="fp64", dt=1e-3),   # more candidates than a group takes
], ids=["big1d", "ragged", "big2d", "scan2", "dense"])
def test_steps_match_oracle(cfg):
    from paper_2501_10965_gb300 import dsmc
    g, o = dsmc.Dsmc(cfg), oracle.OracleSim(cfg)
    g.dsmc_step(3, sample=True)
    o.step(3, sample=True)
    pg, po = _np(g.get_particles()), o.particles()
    assert np.array_equal(pg["cell"], po["cell"])
    for k in KEYS:
        assert np.all(np.abs(pg[k] - po[k]) <= 1e-12 * np.maximum(np.abs(po[k]), 1.0)), k
    for key in ("n_cand", "n_coll", "n_clip", "n_inel", "n_hits"):
        assert g.stats()[key] == o.stats()[key], key
    assert np.allclose(g.accumulators()[0].cpu().numpy(), o.accumulators(), rtol=1e-11, atol=1e-11)


@pytest.mark.parametrize("nx,ny,n", [(5, 1, 700), (5, 1, 20000), (64, 64, 4096), (241, 17, 30001), (130, 95, 1)])
def test_import_keeps_order(nx, ny, n):
    """dsmc_set_particles: sorted by cell, in the given order within a cell."""
    from paper_2501_10965_gb300 import dsmc
    cfg = W.cavity_2d(nx=nx, ny=ny, ppc=1, precision="fp64", capacity=40000)
    g = dsmc.Dsmc(cfg)
    rng = np.random.default_rng(n)
    p = {k: rng.standard_normal(n) for k in KEYS}
    p["x"], p["y"] = rng.uniform(0, 1, n) ** 3, rng.uniform(0, 1, n)
    for _ in range(2):
        g.set_particles({k: torch.tensor(v, device="cuda") for k, v in p.items()})
        out = _np(g.get_particles())
        cell = np.minimum((p["y"] * ny).astype(int), ny - 1) * nx + np.minimum((p["x"] * nx).astype(int), nx - 1)
        order = np.argsort(cell, kind="stable")
        assert np.array_equal(out["cell"], cell[order])
        for k in KEYS:
            assert np.array_equal(out[k], p[k][order]), k
