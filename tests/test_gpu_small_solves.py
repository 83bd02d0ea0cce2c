"""Small networks, whose sums keep one order: whole solves through the
multi-instance runner repeat the recorded states digit by digit (rho, raised
by a quotient of differences at rounding level, loses its ninth digit with any
other order), and the Newton step at the edges of the rule and of the kernels
that only they reach: 400 states, 32 scenarios, 64 rows of K_hat, rows of more
products than a sweep unit holds (a hub), against the oracle at the step bars
without refinement.

golden/small_solves.npz: key "i_seed", the state after the solve to 1e-6 of
instance i with loads of that seed; every `stride`-th entry and the last three
(mu, rho, delta_last)."""
import dataclasses
import os

import numpy as np
import pytest

from bars import step_bars
from oracle import ipm as oipm
from oracle import kkt, opf
from paper_2301_04869_gb300 import synth

pytestmark = pytest.mark.gpu

# buses, generators, scenarios, network seed, stride of the recorded entries
INSTANCES = ((30, 6, 1, 0, 1), (60, 9, 5, 0, 23), (100, 15, 8, 3, 53), (150, 22, 12, 5, 101), (200, 30, 3, 7, 53),
             (120, 18, 17, 9, 101))
SEEDS = (0, 3, 4, 6)


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2301_04869_gb300 import ipm
    ipm.load()
    return ipm


def sample(v, stride):
    return np.r_[v[::stride], v[-3:]]


def solved_states(gpu, seed):
    import torch
    members = []
    for i, (n, ng, N, net_seed, _) in enumerate(INSTANCES):
        net, _, _ = synth.screened_network(n, ng, N, 0.05, seed=net_seed, scen_seed=1)
        pd, qd = synth.make_scenarios(net, N, 0.02, seed=1000 * i + seed)
        members.append(gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64, tol=1e-6))
    _, _, status, _ = gpu.ipm_solve_batch(members)
    assert not status.any()
    out = []
    for sol in members:
        v = torch.empty(sol.dims.state_len, dtype=torch.float64, device="cuda")
        sol.ipm_get_state(v)
        out.append(v.cpu().numpy())
        sol.close()
    return out


@pytest.mark.parametrize("seed", SEEDS)
def test_whole_solves_repeat_recorded_states(gpu, seed):
    want = np.load(os.path.join(os.path.dirname(__file__), "golden", "small_solves.npz"))
    for i, v in enumerate(solved_states(gpu, seed)):
        np.testing.assert_array_equal(sample(v, INSTANCES[i][4]), want[f"{i}_{seed}"], err_msg=str(INSTANCES[i]))


def hub(net, extra):
    """`extra` more lines from the last bus, with the first lines' constants."""
    last = net.n_bus - 1
    near = np.r_[net.to[net.fr == last], net.fr[net.to == last], last]
    to = np.setdiff1d(np.arange(net.n_bus), near)[:extra].astype(net.to.dtype)
    return dataclasses.replace(
        net, fr=np.r_[net.fr, np.full(extra, last, net.fr.dtype)], to=np.r_[net.to, to],
        **{k: np.r_[getattr(net, k), getattr(net, k)[:extra]] for k in ("r", "x", "b")})


# buses, generators, scenarios, extra lines of a hub
EDGES = [(5, 2, 1, 0), (60, 9, 31, 0), (60, 9, 32, 0), (60, 9, 33, 0), (216, 32, 2, 0), (216, 31, 2, 0), (216, 30, 2, 0),
         (216, 33, 1, 0), (180, 32, 1, 0), (80, 10, 3, 40), (190, 20, 2, 150)]


@pytest.mark.parametrize("n,ng,N,extra", EDGES)
def test_step_at_the_edges_of_the_small_problems(gpu, n, ng, N, extra):
    import torch
    net = synth.make_network(n, ng, seed=3)
    if extra:
        net = hub(net, extra)
    pd, qd = synth.make_scenarios(net, N, 0.05, seed=4)
    M = opf.Model(net, pd, qd)
    st = oipm.initial_state(M)
    D = kkt.eval_all(M, st)
    C, L, delta = oipm.factor_with_inertia_correction(M, dict(st), D, st["mu"])
    p = kkt.reduced_step(M, st, D, C, L)
    sol = gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64, aug_refine=0)
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    assert sol.ipm_factor_schur(delta)
    step = torch.empty(sol.dims.step_len, dtype=torch.float64, device="cuda")
    sol.ipm_solve_kkt(step)
    g = sol.split_step(step.cpu().numpy())
    bars = step_bars(M, st, D, C, p)
    for k in ("px", "pu", "ps", "py", "pz"):
        err = np.abs(g[k] - p[k]).max() / max(np.abs(p[k]).max(), 1e-300)
        assert err <= bars[k], (k, err, bars[k])
    sol.close()
