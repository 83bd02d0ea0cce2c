"""Device memory of the multi-RHS solve's work buffer: the panels of the CTAs
that are on the GPU at once (760 of 256 threads, 32 columns each with a large
trailing block), in the type of the path, whatever the number of scenarios.

Everything else in a context of one network grows in proportion to the
scenarios, and so does the buffer until it holds its 760 panels (29 panels per
scenario on this network: from 27 scenarios on), so two small and two large
contexts give its size at the large ones.  On the mixed path the small contexts'
buffer is for the FP64 solve of a fallback iteration, the large ones' for the
FP32 solve (the FP64 one then fits the operands' region).  Half of the buffer is
left for the rounding of the allocations."""
import pytest

from paper_2301_04869_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2301_04869_gb300 import ipm
    ipm.load()
    return ipm


@pytest.mark.parametrize("precision,elem", [("fp64", 8), ("mixed", 4)])
def test_work_buffer_is_bounded(gpu, precision, elem):
    import torch
    net = synth.make_network(3000, 450, seed=0, load_scale=0.3)
    pd, qd = synth.make_scenarios(net, 72, 0.05, seed=1)
    prec = gpu.PREC_FP64 if precision == "fp64" else gpu.PREC_MIXED

    def used(n):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        sol = gpu.Solver(net, pd[:n], qd[:n], precision=prec)
        nx, nu = sol.dims.n_x, sol.dims.n_u
        mem = before - torch.cuda.mem_get_info()[0]
        sol.close()
        return mem, nx, nu

    used(2)  # what the first context leaves behind
    (m8, nx, nu), m24, m56, m72 = used(8), used(24)[0], used(56)[0], used(72)[0]
    assert (nx, nu) == (5549, 899)
    small, large = (m24 - m8) / 16, (m72 - m56) / 16  # per scenario, the buffer growing and at its size
    buffer = m56 - 56 * large - (m8 - 8 * small)
    assert buffer <= 1.5 * 760 * nx * 32 * elem, (buffer / 2**20, small / 2**20, large / 2**20)
