"""FP32 layout: the launches of a call follow one another with nothing between
them, whatever the number of steps, so that the launch shapes that a first
long call times are timed alike."""
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu



def _traced(call):
    """names of the kernels and memory operations of the call, in order"""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    ev = [e for e in prof.events() if "dsmc::" in e.name or e.name.startswith("Mem")]
    return [e.name for e in sorted(ev, key=lambda e: e.time_range.start)]


@pytest.mark.parametrize("nsteps", [1, 6, 20, 21, 25])
def test_no_clear_between_the_launches_of_a_call(nsteps):
    from paper_2501_10965_gb300 import dsmc
    g = dsmc.Dsmc(W.homogeneous_box(ncells=40, ppc=60, dt=4e-3, precision="fp32"))
    _traced(lambda: g.num_particles())  # a process's first trace may stay empty
    names = _traced(lambda: g.dsmc_step(nsteps))
    if not any("dsmc::" in n for n in names):
        pytest.skip("no kernel trace here")
    assert all("fused" in n for n in names[:nsteps]), names[:nsteps]
    assert "collide" in names[nsteps] and not any("Memset" in n for n in names)
    assert g.stats()["n_overflow"] == 0 and g.num_particles() == 40 * 60
