"""1D synthetic solve: above 304 slabs a slab takes half the threads; the
solutions are those of a handle at the line (reductions in another order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(40, 128), (129, 256), (257, 300)])
def test_slabs_on_both_sides_of_the_line(sizes):
    from paper_2501_10965_gb300 import dsmc
    cases = [W.fourier_1d(nx=sizes[i % 2], ppc=40, seed=i, precision="fp32", synth_tol=1e-13, n_m=60)
             for i in range(305)]
    g, h = dsmc.Dsmc(cases), dsmc.Dsmc(cases[:304])
    g.dsmc_step(40, sample=True)
    f = g.dsmc_sample(reset=False)
    hot, _, _ = g.dsmc_hot(f)
    n = sum(c["nx"] for c in cases[:304])
    # a slab whose noisy HoT admits no solution keeps its sampled fields, on either side
    a = g.synth_solve(f, hot, allow_fallback=True)[0][:n].cpu().numpy()
    b = h.synth_solve(f[:n].contiguous(), hot[:n].contiguous(), allow_fallback=True)[0].cpu().numpy()
    np.testing.assert_allclose(a, b, rtol=1e-9, atol=1e-11)
