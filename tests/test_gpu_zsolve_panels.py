"""The multi-RHS solve at the edges of its panels (8, 16 or 32 columns, chosen
from n_u and the number of scenarios; b = G_x^{-1} g in the last panel's free
place): n_u + 1 just filling a panel and one past it, few scenarios and many,
against the oracle at the cold start.  Bars as elsewhere: FP64 1e-10, mixed
(FP32 solve, BF16x3 contraction) 1e-5, both normwise, the reduced right-hand
side 1e-10 on both."""
import numpy as np
import pytest

from oracle import ipm as oipm
from oracle import kkt, opf
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


def rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


# generators n_g (n_u + 1 = 2 n_g columns) and scenarios
@pytest.mark.parametrize("ng,N", [(4, 2), (5, 1), (16, 2), (17, 3), (16, 40), (17, 40), (16, 152), (17, 160)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_panel_edges(gpu, ng, N, precision):
    net = synth.make_network(47, ng, seed=3)
    pd, qd = synth.make_scenarios(net, N, 0.05, seed=4)
    M = opf.Model(net, pd, qd)
    st = oipm.initial_state(M)
    C = kkt.condense(M, st, kkt.eval_all(M, st), st["mu"], 0.0)
    sol = gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64 if precision == "fp64" else gpu.PREC_MIXED)
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    nx, nu = sol.dims.n_x, sol.dims.n_u
    bar = 1e-10 if precision == "fp64" else 1e-5
    assert rel(sol.ipm_get_quantity(gpu.Q_KHAT).reshape(nu, nu), C.Khat) <= bar
    assert rel(sol.ipm_get_quantity(gpu.Q_RHS_U), C.rhs_u) <= 1e-10
    for i in (0, N - 1):
        assert rel(sol.ipm_get_quantity(gpu.Q_Z, i).reshape(nx, nu), C.Z[i]) <= bar, i
