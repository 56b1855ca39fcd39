"""Particle modification of the FP32 layout, cell by cell at the sizes where
the register path's parts change (one lane, a warp's edges, its limit of 256
and above it), with removals, additions, both velocity scales and copies of
one particle: the result is the FP32 rounding of the FP64 linear map."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu

#        before, after
COUNTS = [(1, 1), (1, 40), (2, 1), (31, 31), (32, 32), (33, 32), (64, 65), (100, 60), (200, 215), (255, 256), (256, 256),
          (256, 3), (250, 257), (257, 256), (300, 310)]


@pytest.mark.parametrize("scale,same", [(1.0, False), (300.0, False), (1e-3, False), (1.0, True)])
@pytest.mark.parametrize("dim", [1, 2])
def test_linear_map_and_counts(dim, scale, same):
    from paper_2501_10965_gb300 import dsmc
    nx = len(COUNTS)
    kw = dict(precision="fp32", capacity=40000, ppc=200, kn=0.1)
    cfg = W.base_config(dim=1, nx=nx, **kw) if dim == 1 else W.base_config(dim=2, nx=nx, ny=1, **kw)
    g = dsmc.Dsmc(cfg)
    rng = np.random.default_rng(3)
    n0 = [a for a, _ in COUNTS]
    x = np.concatenate([(c + rng.uniform(0.01, 0.99, n)) / nx for c, n in enumerate(n0)])
    n = len(x)
    p = {"x": x, "y": rng.uniform(0.1, 0.9, n) if dim == 2 else np.zeros(n), "vx": scale * (rng.standard_normal(n) + 0.3),
         "vy": scale * rng.standard_normal(n), "vz": scale * (rng.standard_normal(n) - 2.0), "ir": scale * rng.exponential(size=n)}
    if same:
        for k in ("vx", "vy", "vz", "ir"):
            p[k][:] = p[k][0]
    g.set_particles({k: torch.tensor(v, device="cuda") for k, v in p.items()})
    src = {k: v.cpu().numpy() for k, v in g.get_particles().items()}
    fnum = g.constants()["fnum"]
    tgt = np.zeros((nx, 6))
    tgt[:, 0] = np.array([b for _, b in COUNTS]) * fnum * nx
    tgt[:, 1:4] = np.array([0.1, -0.2, 0.05]) * scale
    tgt[:, 4] = 1.1 * scale ** 2
    tgt[:, 5] = 0.9 * scale
    g.dig_correct(torch.tensor(tgt, device="cuda"))
    out = {k: v.cpu().numpy() for k, v in g.get_particles().items()}
    for c, (na, nb) in enumerate(COUNTS):
        a, b = src["cell"] == c, out["cell"] == c
        assert a.sum() == na and abs(int(b.sum()) - nb) <= 1  # Iround at an integer up to FP64 rounding
        nb = int(b.sum())
        s = {k: src[k][a] for k in src}
        o = {k: out[k][b] for k in out}
        kept = min(na, nb)
        # kept particles keep their place and order; the others lie in the cell
        at = {v: i for i, v in enumerate(s["x"])}
        idx = [at[v] for v in o["x"][:kept]]
        assert idx == sorted(idx) and len(set(idx)) == kept
        assert np.all((o["x"] >= c / nx - 1e-6) & (o["x"] <= (c + 1) / nx + 1e-6))
        assert np.array_equal(o["y"][:kept], s["y"][idx])
        new = {}
        for k in ("vx", "vy", "vz", "ir"):
            new[k] = s[k][idx].astype(np.float64)
        if nb > na:
            # the copies: each one is the image of a source particle; find it by I_r
            # after the map is known up to the copies themselves, so test the moments
            for q, t in ((1, "vx"), (2, "vy"), (3, "vz")):
                assert abs(o[t].mean() - tgt[c, q]) <= 1e-6 * scale * 4
            assert abs(o["ir"].mean() - tgt[c, 5]) <= 1e-6 * scale * 4
            continue
        u = [new[k].mean() for k in ("vx", "vy", "vz")]
        tts = sum(((new[k] - u[q]) ** 2).sum() for q, k in enumerate(("vx", "vy", "vz"))) / (3.0 * nb)
        fa = np.sqrt(tgt[c, 4] / tts) if nb >= 2 and tts > 1e-20 * scale ** 2 else 1.0
        fc = tgt[c, 5] / new["ir"].mean()
        for q, k in enumerate(("vx", "vy", "vz")):
            want = fa * new[k] + (tgt[c, 1 + q] - fa * u[q])
            ulp = np.spacing(np.maximum(np.abs(want), 1e-30).astype(np.float32)).astype(np.float64)
            # half an ulp of the rounding plus FP64 rounding of a and b
            assert np.all(np.abs(o[k] - want) <= 0.5001 * ulp + 1e-13 * scale * (1 + fa)), (c, k)
        want = fc * new["ir"]
        ulp = np.spacing(want.astype(np.float32)).astype(np.float64)
        assert np.all(np.abs(o["ir"] - want) <= 0.5001 * ulp + 1e-13 * scale)


@pytest.mark.parametrize("nx,ny", [(64, 64), (4097, 1), (123, 100)])
def test_scan_over_the_grid(nx, ny):
    """Counts and offsets of the modification and the read-out beyond one CTA."""
    from paper_2501_10965_gb300 import dsmc
    cfg = W.base_config(dim=2, nx=nx, ny=ny, ppc=3, precision="fp32")
    g = dsmc.Dsmc(cfg)
    tgt = np.zeros((nx * ny, 6))
    tgt[:, 0] = 1.0 + (np.arange(nx * ny) % 5) * 0.34
    tgt[:, 4:] = 1.0
    g.dig_correct(torch.tensor(tgt, device="cuda"))
    p = g.get_particles()
    cnt = np.bincount(p["cell"].cpu().numpy(), minlength=nx * ny)
    assert np.all(np.abs(cnt - 3.0 * tgt[:, 0]) < 1.0 + 1e-9) and cnt.sum() == g.num_particles()
    cell = p["cell"].cpu().numpy()
    assert np.all(np.diff(cell) >= 0)
    # positions lie in their cell up to the rounding of an FP32 position at an edge
    for axis, n, i in (("x", nx, cell % nx), ("y", ny, cell // nx)):
        v = p[axis].cpu().numpy()
        assert np.all((v >= i / n - 3e-7) & (v <= (i + 1) / n + 3e-7))
