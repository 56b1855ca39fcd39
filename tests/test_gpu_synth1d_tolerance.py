"""1D synthetic solve: the largest relative update of a Newton step, which is
compared with the tolerance, is an FP64 number.  It is found here by bisection
over the tolerance and formed from the iterates."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _inputs(nx):
    x = (np.arange(nx) + 0.5) / nx
    f = np.zeros((nx, 18))
    f[:, 0] = 1.0 + 0.1 * np.cos(np.pi * x)
    f[:, 2], f[:, 3] = 0.2 * np.sin(2.0 * x), 0.1 * x
    f[:, 4], f[:, 5] = 1.0 + 0.2 * x, 1.0 + 0.15 * x ** 2
    h = np.zeros((nx, 12))
    h[:, 0], h[:, 3], h[:, 6], h[:, 9] = (a * np.sin(k * x) for a, k in ((1e-3, 5), (2e-3, 3), (1e-3, 4), (1e-3, 6)))
    return (torch.tensor(a, device="cuda") for a in (f, h))


@pytest.mark.parametrize("nx,step", [(40, 2), (200, 2), (200, 3)])
def test_step_size_against_the_tolerance(nx, step):
    from paper_2501_10965_gb300 import dsmc
    f, h = _inputs(nx)

    def solve(tol, n_m):
        g = dsmc.Dsmc(W.couette_1d(nx=nx, ppc=2, precision="fp64", synth_tol=tol, n_m=n_m))
        out, it, _ = g.synth_solve(f, h, allow_not_converged=True, allow_fallback=True)
        assert g.last_synth_status in (0, -4)
        return out.cpu().numpy(), it

    y0, y1 = (solve(1e-300, step - k)[0] for k in (1, 0))
    cols = [2, 3, 4, 5]  # the unknowns u_y, u_z, T_t, T_r
    d = np.abs(y1[:, cols] - y0[:, cols]) / np.maximum(np.abs(y0[:, cols]), 1e-3)
    # the pressure's step, from P = rho T_t + HoT_xx, must not decide here
    P = [(y[:, 0] * y[:, 4] + h[:, 0].cpu().numpy()).mean() for y in (y0, y1)]
    assert abs(P[1] - P[0]) / abs(P[0]) < 0.5 * d.max()
    # the smallest tolerance that ends the iteration at this step
    lo, hi = d.max() * (1 - 1e-5), d.max() * (1 + 1e-5)
    assert solve(lo, step + 1)[1] == step + 1 and solve(hi, step + 1)[1] == step
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        if solve(mid, step + 1)[1] == step:
            hi = mid
        else:
            lo = mid
    # the same numbers, one subtraction and one division: equal but for the
    # bisection's last interval, 2e-5 2^-40
    assert abs(hi / d.max() - 1) <= 1e-14
