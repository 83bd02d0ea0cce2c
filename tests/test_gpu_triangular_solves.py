"""The single-vector solves at the edges of their blocks: trailing blocks of
G_x just below, at and above one and two diagonal blocks (32 rows in one CTA,
64 in the cluster kernel of the large blocks, forced here), and K_hat at the
sizes where its solve goes from one CTA to a cluster and from 32 to 64 rows.
The Newton step at the cold start against the oracle at the step bars, on the
FP64 path without refinement (the transposed solve and the Cholesky solve, and
with a large block the forward solve, as they are) and on the mixed path (both
solves in every product of the conjugate gradients)."""
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


def rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


# (buses, generators, scenarios, large-block kernels, states of the trailing block or None)
EDGES = [(160, 22, 2, False, 31), (190, 27, 1, False, 32), (181, 25, 3, False, 33), (372, 53, 1, False, 64),
         (374, 53, 2, False, 65), (214, 30, 1, True, 63), (183, 26, 2, True, 64), (178, 25, 39, True, 65),
         (406, 58, 1, True, 128), (350, 50, 2, True, 129),
         (300, 64, 1, False, None), (300, 65, 2, False, None), (300, 256, 1, False, None), (300, 257, 1, False, None)]
DELTA = {256: 100.0}  # inertia correction where K_hat of the cold start is indefinite


@pytest.mark.parametrize("n,ng,N,big,nd", EDGES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_step_at_block_edges(gpu, n, ng, N, big, nd, precision):
    import torch
    net = synth.make_network(n, ng, seed=3)
    pd, qd = synth.make_scenarios(net, N, 0.05, seed=4)
    M = opf.Model(net, pd, qd)
    st = oipm.initial_state(M)
    D = kkt.eval_all(M, st)
    delta = DELTA.get(ng, 0.0)
    C = kkt.condense(M, st, D, st["mu"], delta)
    p = kkt.reduced_step(M, st, D, C, kkt.cholesky_pd(C.Khat))
    kw = dict(precision=gpu.PREC_FP64, aug_refine=0) if precision == "fp64" else dict(precision=gpu.PREC_MIXED)
    sol = gpu.Solver(net, pd, qd, big_block=big, **kw)
    assert nd is None or sol.dims.nd == nd
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    assert sol.ipm_factor_schur(delta)
    step = torch.empty(sol.dims.step_len, dtype=torch.float64, device="cuda")
    sol.ipm_solve_kkt(step)
    g = sol.split_step(step.cpu().numpy())
    bars = step_bars(M, st, D, C, p)
    for k in ("px", "pu", "ps", "py", "pz"):
        assert rel(g[k], p[k]) <= bars[k], (k, rel(g[k], p[k]), bars[k])
