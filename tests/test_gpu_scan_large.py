"""The scan over the grid beyond one piece of 4 096 cells per SM (622 592 cells),
where a CTA passes over several pieces: counts and offsets of the modification
and the read-out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(4096, 152), (811, 773), (4096, 305), (1999, 1001)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_scan_of_several_pieces(nx, ny, precision):
    from paper_2501_10965_gb300 import dsmc
    n = nx * ny
    g = dsmc.Dsmc(W.base_config(dim=2, nx=nx, ny=ny, ppc=2, precision=precision))
    want = np.arange(n) % 5
    want[want == 0] = 2
    tgt = np.zeros((n, 6))
    # rho V / F is the wanted count up to FP64 rounding, which Iround all but never sees
    tgt[:, 0] = want / 2.0
    tgt[:, 4:] = 1.0
    g.dig_correct(torch.tensor(tgt, device="cuda"))
    assert g.num_particles() == want.sum()
    cell = g.get_particles()["cell"]
    assert torch.equal(torch.bincount(cell, minlength=n), torch.tensor(want, device="cuda"))
    assert bool((cell[1:] >= cell[:-1]).all())
