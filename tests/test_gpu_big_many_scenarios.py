"""The large-block kernels where their choices hang on the number of scenarios
(forced on small networks): the rows of U by a thread per column from 304
column tiles on (two tiles of the first panel at 153 and 160 scenarios, the
last ragged; by a warp per column below), the sparse part by clusters of four,
two CTAs or one per scenario (up to 76, 152, more), and the adjoint reduction's
solves through a large block by one CTA per vector.  Z, K_hat and the reduced
right-hand side at the cold start against the oracle at 1e-10."""
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


# buses, generators, scenarios, states of the trailing block, adjoint reduction
CASES = [(350, 50, 160, 129, False), (350, 50, 153, 129, False), (350, 50, 152, 129, False), (183, 26, 77, 64, False),
         (183, 26, 76, 64, False), (350, 50, 3, 129, True)]


@pytest.mark.parametrize("n,ng,N,nd,adjoint", CASES)
def test_condensation(gpu, n, ng, N, nd, adjoint):
    net = synth.make_network(n, ng, seed=3)
    pd, qd = synth.make_scenarios(net, N, 0.05, seed=4)
    M = opf.Model(net, pd, qd)
    st = oipm.initial_state(M)
    C = kkt.condense(M, st, kkt.eval_all(M, st), st["mu"], 0.0)
    sol = gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64, big_block=True,
                     reduction=gpu.REDUCTION_ADJOINT if adjoint else gpu.REDUCTION_DENSE)
    assert sol.dims.nd == nd and sol.dims.big_block
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    pairs = [(sol.ipm_get_quantity(gpu.Q_KHAT), C.Khat), (sol.ipm_get_quantity(gpu.Q_RHS_U), C.rhs_u)]
    pairs += [(sol.ipm_get_quantity(gpu.Q_Z, i), C.Z[i]) for i in sorted({0, N // 2, N - 1})]
    for got, want in pairs:
        assert np.abs(got.reshape(want.shape) - want).max() <= 1e-10 * np.abs(want).max()
    sol.close()
