"""2D synthetic solve: the panel kernel that also applies the panel before it,
at the heights (kl + 32, kl = 10 min(nx, ny) + 4) where its form changes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import synth2d
from oracle.fields import F_RHO
from test_gpu_synth2d import _cfg, _dev, _gpu, _smooth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [
    (31, 3),     # 66 rows: fewer threads than a panel's columns take warps, a ragged last panel
    (35, 36),    # 386 rows: above 384 threads
    (98, 98),    # 1 016 rows: a row a thread, the tallest such
    (99, 99),    # 1 026: two rows a thread
    (124, 125),  # 1 276: the tallest of two rows
    (125, 125),  # 1 286: three rows
    (151, 151),  # 1 546: panels in shared memory, but for the last ones
])
def test_solution_satisfies_the_oracle_equations(nx, ny):
    """As at full size: converged, the oracle's residual below 1e-9 at every
    cell (against O(100) terms), the total mass kept to 1e-12."""
    cfg = _cfg(nx, ny, ppc=2, synth_tol=1e-10)
    d, h = _smooth(nx, ny, seed=5)
    out, it, res = _gpu(cfg).synth_solve(_dev(d), _dev(h))
    assert res < 1e-9 and it <= 10
    o = out.cpu().numpy()
    r = synth2d.residual(np.concatenate([o[:, 0], o[:, 1], o[:, 2], o[:, 4], o[:, 5]]), d, h, cfg)
    assert np.max(np.abs(r)) < 1e-9
    assert abs(o[:, 0].sum() / d[:, F_RHO].sum() - 1.0) < 1e-12
