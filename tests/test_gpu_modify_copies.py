"""Particle modification of the FP32 layout: copies of one particle have no
thermal spread, whatever the sizes of its velocity components, so each of them
takes the target velocity; and a component much smaller than the others keeps
its digits."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu

#        before, after
COUNTS = [(1, 2), (1, 40), (1, 256), (1, 300), (40, 40), (100, 60), (100, 215), (256, 256), (300, 280)]
TARGET = (0.1, -0.2, 0.05)


def _modified(vel, ir, seed):
    """the cells' particles before and after; vel(n): n x 3"""
    from paper_2501_10965_gb300 import dsmc
    nx = len(COUNTS)
    g = dsmc.Dsmc(W.base_config(dim=1, nx=nx, precision="fp32", capacity=40000, ppc=200, kn=0.1))
    rng = np.random.default_rng(seed)
    n0 = [a for a, _ in COUNTS]
    x = np.concatenate([(c + rng.uniform(0.01, 0.99, n)) / nx for c, n in enumerate(n0)])
    v = vel(rng, len(x))
    p = {"x": x, "y": 0 * x, "vx": v[:, 0], "vy": v[:, 1], "vz": v[:, 2], "ir": ir(rng, len(x))}
    g.set_particles({k: torch.tensor(q, device="cuda") for k, q in p.items()})
    src = {k: q.cpu().numpy() for k, q in g.get_particles().items()}
    tgt = np.zeros((nx, 6))
    tgt[:, 0] = np.array([b for _, b in COUNTS]) * g.constants()["fnum"] * nx
    tgt[:, 1:4] = TARGET
    tgt[:, 4], tgt[:, 5] = 1.1, 0.9
    g.dig_correct(torch.tensor(tgt, device="cuda"))
    out = {k: q.cpu().numpy() for k, q in g.get_particles().items()}
    for c in range(nx):
        a, b = src["cell"] == c, out["cell"] == c
        yield {k: src[k][a] for k in src}, {k: out[k][b] for k in out}


@pytest.mark.parametrize("v", [(1.0, 1e-7, 0.3), (5.0, 1e-6, 2.0), (1.3, -0.7, 3.1234567e-8), (0.1, 0.1, 0.1),
                               (3e6, -1e-38, 0.25), (3e18, 1e-44, 1e-6)])
def test_copies_take_the_target_velocity(v):
    """a = 1, so each copy becomes v + (target - v): FP64 rounds the two sums by
    2^-53 (|v| + |target|) each at most, and the result to 32 bits once."""
    for s, o in _modified(lambda rng, n: np.tile(v, (n, 1)), lambda rng, n: np.full(n, 0.7), 5):
        assert len(o["x"]) >= 2
        for q, k in enumerate(("vx", "vy", "vz")):
            assert np.all(s[k] == s[k][0])
            t = TARGET[q]
            tol = 0.5 * float(np.spacing(np.float32(abs(t)))) + 2.0 ** -52 * (abs(s[k][0]) + abs(t))
            assert np.all(np.abs(o[k] - t) <= tol), (k, len(s[k]), len(o[k]), o[k][:4])


@pytest.mark.parametrize("small", [1e-5, 1e-8, 1e-20])
def test_a_small_component_keeps_its_digits(small):
    """Cells that keep their particles: the map of the FP64 moments, rounded to
    32 bits once.  a carries a relative FP64 error of some 2^-50 (256 terms), and
    b the error of a times the mean."""
    scale = np.array([1.0, small, 0.3])
    vel = lambda rng, n: rng.standard_normal((n, 3)) * scale
    for s, o in _modified(vel, lambda rng, n: rng.exponential(size=n), 6):
        n = len(s["x"])
        if len(o["x"]) != n or n < 2:
            continue
        names = ("vx", "vy", "vz")
        u = [math.fsum(s[k]) / n for k in names]
        tts = math.fsum(((s[k] - u[q]) ** 2).sum() for q, k in enumerate(names)) / (3.0 * n)
        a = math.sqrt(1.1 / tts)
        for q, k in enumerate(names):
            want = a * (s[k] - u[q]) + TARGET[q]
            tol = 0.5001 * np.spacing(np.abs(want).astype(np.float32)).astype(np.float64) + 2.0 ** -49 * (
                a * np.abs(s[k]) + a * abs(u[q]) + abs(TARGET[q]))
            assert np.all(np.abs(o[k] - want) <= tol), (k, n)
