"""The Newton step late in a solve, where K_hat and the G_x blocks are worst
conditioned, without refinement: the single-vector solves and the Cholesky
solve by inverted diagonal blocks (more than 400 states, more than 64 rows of
K_hat; 64-row blocks with a large trailing block) and by substitution (the
smaller ones): p_u and p_x against the oracle at the step bars (10 kappa eps,
around 1e-3 there; the recovered blocks' bars pass 1 and say nothing)."""
import numpy as np
import pytest

from bars import step_bars
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


@pytest.mark.parametrize("n,ng,N,big", [(120, 18, 5, False), (300, 45, 2, False), (433, 65, 3, False), (433, 65, 3, True)])
def test_late_step(gpu, n, ng, N, big):
    import torch
    net, pd, qd = synth.screened_network(n, ng, N, 0.05, seed=3, scen_seed=4)
    M = opf.Model(net, pd, qd)
    sol = gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64, aug_refine=0, big_block=big, tol=1e-6)
    sol.ipm_solve()
    st = sol.split_state(sol.ipm_get_state())
    D = kkt.eval_all(M, st)
    C, L, delta = oipm.factor_with_inertia_correction(M, dict(st), D, st["mu"])
    p = kkt.reduced_step(M, st, D, C, L)
    bars = step_bars(M, st, D, C, p)
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    assert sol.ipm_factor_schur(delta)
    step = torch.empty(sol.dims.step_len, dtype=torch.float64, device="cuda")
    sol.ipm_solve_kkt(step)
    g = sol.split_step(step.cpu().numpy())
    for k in ("px", "pu"):
        err = np.abs(g[k] - p[k]).max() / np.abs(p[k]).max()
        assert err <= bars[k] < 1e-2, (k, err, bars[k])
    sol.close()
