"""FP64 layout: steps captured into a CUDA graph run on whatever particles the
handle holds when the graph is launched, also those that dsmc_set_particles or
dig_correct put there after the capture."""
import pytest

torch = pytest.importorskip("torch")

from paper_2501_10965_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NSTEPS = 2  # even: a captured call finds the buffers where it left them


def _same(a, b):
    pa, pb = a.get_particles(), b.get_particles()
    assert a.num_particles() == b.num_particles() > 0
    for k in pa:
        assert torch.equal(pa[k], pb[k]), k


@pytest.mark.parametrize("between", ["nothing", "set_particles", "dig_correct"])
@pytest.mark.parametrize("ncells", [7, 700])  # scan and lists in one CTA, or over the grid
def test_captured_steps_see_new_particles(ncells, between):
    from paper_2501_10965_gb300 import dsmc
    cfg = W.homogeneous_box(ncells=ncells, ppc=30, dt=4e-3, precision="fp64", kn=0.1)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a, b = dsmc.Dsmc(cfg, stream=st), dsmc.Dsmc(cfg, stream=st)
        for g in (a, b):
            g.dsmc_step(NSTEPS)
        graph = torch.cuda.CUDAGraph()
        p = a.get_particles()
        with torch.cuda.graph(graph, stream=st):
            a.dsmc_step(NSTEPS)
        for g in (a, b):  # twice: the buffers are where they were at the capture
            for _ in range(2):
                if between == "set_particles":
                    g.set_particles(p)
                elif between == "dig_correct":
                    t = torch.zeros(ncells, 6, dtype=torch.float64, device="cuda")
                    t[:, 0], t[:, 4:] = 1.0, 1.0
                    g.dig_correct(t)
        graph.replay()
        b.dsmc_step(NSTEPS)
        st.synchronize()
        _same(a, b)
        graph.replay()
        b.set_counters(NSTEPS, b.counters()[1])  # the graph repeats its steps' numbers
        b.dsmc_step(NSTEPS)
        st.synchronize()
        _same(a, b)
