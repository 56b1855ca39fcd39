"""FP32 layout, handles with few cells: the fused step with a CTA per cell is
among the launch shapes that a first call of at least 20 steps times, so such
a call runs it for four steps at least.  Checked where it changes form: cells
above its tile, bins that overflow, few particles, 2D, a batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NSTEPS = 25  # one launch more than four shapes' sixteen and the odd first ones
SPEC = [{"kind": "specular", "T": 1, "u": (0, 0, 0)}] * 4


def _np(p):
    return {k: v.cpu().numpy() for k, v in p.items()}


def _box2d(**kw):
    cfg = W.base_config(dim=2, walls=SPEC, precision="fp32", dt=4e-3)
    cfg.update(kw)
    return cfg


def _crowd(cfg, cell, n):
    """cfg's own cells of ppc particles, and n in one cell"""
    rng = np.random.default_rng(11)
    nx, ny = cfg["nx"], cfg["ny"]
    per = np.full(nx * ny, cfg["ppc"])
    per[cell] = n
    c = np.repeat(np.arange(nx * ny), per)
    m = len(c)
    p = {"x": (c % nx + rng.random(m)) / nx, "y": (c // nx + rng.random(m)) / ny * (cfg["dim"] == 2)}
    p.update({k: rng.standard_normal(m) for k in ("vx", "vy", "vz")}, ir=rng.exponential(1.0, m))
    return {k: torch.tensor(v) for k, v in p.items()}


CASES = {
    "small": (W.homogeneous_box(ncells=3, ppc=5, dt=4e-3, precision="fp32"), None),
    "crowd": (W.homogeneous_box(ncells=12, ppc=60, dt=4e-3, precision="fp32", capacity=20000), (5, 2100)),
    "tight": (W.homogeneous_box(ncells=40, ppc=200, dt=4e-3, precision="fp32", bin_slack=1.0, init_u=(2.0, 0.0, 0.0)),
              None),
    "2d": (_box2d(nx=17, ny=9, ppc=50), None),
    "crowd2d": (_box2d(nx=8, ny=8, ppc=40, capacity=40000), (63, 1500)),
    "batch": ([W.homogeneous_box(ncells=c, ppc=n, dt=4e-3, precision="fp32", seed=c)
               for c, n in ((7, 30), (40, 200), (21, 64))], None),
    "batch2d": ([_box2d(nx=6, ny=5, ppc=n, seed=n) for n in (20, 90)], None),
}


def _start(name, **kw):
    from paper_2501_10965_gb300 import dsmc
    cfg, crowd = CASES[name]
    cfg = [dict(c, **kw) for c in cfg] if isinstance(cfg, list) else dict(cfg, **kw)
    g = dsmc.Dsmc(cfg)
    if crowd:
        g.set_particles(_crowd(cfg, *crowd))
    return g, cfg if isinstance(cfg, list) else [cfg]


@pytest.mark.parametrize("name", CASES)
def test_free_flight_between_specular_walls(name):
    """Without collisions every particle's path is known: x folded into the
    box, its velocity's sign with it.  Particles are told apart by vz.  A step
    rounds a position at most four times (product, sum, reflection) by 2^-24 of
    a coordinate below 2: NSTEPS 4 2^-23 < 1.2e-5 in all."""
    g, cfgs = _start(name, kn=1e12)
    a = _np(g.get_particles())
    g.dsmc_step(NSTEPS, sample=True)
    b = _np(g.get_particles())
    assert len(a["x"]) == len(b["x"])
    assert g.launch_shape() != (0, 0)
    cell0 = np.concatenate([[0], np.cumsum([c["nx"] * c["ny"] for c in cfgs])])
    for k, cfg in enumerate(cfgs):
        A, B = ({q: v[(p["cell"] >= cell0[k]) & (p["cell"] < cell0[k + 1])] for q, v in p.items()} for p in (a, b))
        ia, ib = (np.lexsort((p["ir"], p["vz"])) for p in (A, B))
        assert np.array_equal(A["vz"][ia], B["vz"][ib]) and np.array_equal(A["ir"][ia], B["ir"][ib])
        for x, v in (("x", "vx"), ("y", "vy"))[: cfg["dim"]]:
            t = A[x][ia] + A[v][ia] * cfg["dt"] * NSTEPS
            f = np.mod(t, 2.0)
            assert np.all(np.abs(np.where(f > 1.0, 2.0 - f, f) - B[x][ib]) <= 1.2e-5)
            assert np.array_equal(np.abs(A[v][ia]), np.abs(B[v][ib]))
    # every particle sampled once a step, unless it waits on the overflow list
    # (a lane adds at most 66 particles at a time in FP32)
    acc, waits = g.accumulators()[0].cpu().numpy(), g.stats()["n_overflow"]
    assert acc[:, 0].sum() + waits == NSTEPS * len(a["x"])
    if waits == 0:
        assert abs(acc[:, 3].sum() - NSTEPS * a["vz"].sum()) <= 2e-6 * NSTEPS * np.abs(a["vz"]).sum()
    if name == "tight":
        assert waits > 0


@pytest.mark.parametrize("name", CASES)
def test_collisions_conserve(name):
    """Momentum along z and energy stay: a collision rounds each velocity by
    a few 2^-24, here some ten collisions a particle."""
    g, cfgs = _start(name, kn=0.01)
    a = _np(g.get_particles())
    g.dsmc_step(NSTEPS, sample=True)
    b = _np(g.get_particles())
    assert len(a["x"]) == len(b["x"]) and g.stats()["n_coll"] > 0
    cell0 = np.concatenate([[0], np.cumsum([c["nx"] * c["ny"] for c in cfgs])])
    for k in range(len(cfgs)):
        A, B = ({q: v[(p["cell"] >= cell0[k]) & (p["cell"] < cell0[k + 1])] for q, v in p.items()} for p in (a, b))
        assert abs(A["vz"].sum() - B["vz"].sum()) <= 1e-5 * np.abs(A["vz"]).sum()
        e = [(0.5 * (p["vx"] ** 2 + p["vy"] ** 2 + p["vz"] ** 2) + p["ir"]).sum() for p in (A, B)]
        assert abs(e[1] - e[0]) <= 1e-5 * e[0]
    assert g.accumulators()[0].cpu().numpy()[:, 0].sum() + g.stats()["n_overflow"] == NSTEPS * len(a["x"])
