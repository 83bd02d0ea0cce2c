"""The model functions and their derivatives where a (bus, scenario) pair goes
from eight lanes to one (24,320 pairs): both forms add a bus's lines in the
same order, so a scenario's functions and Jacobians are the same to the last
bit below, at and above the switch."""
import numpy as np
import pytest

from oracle import ipm as oipm
from oracle import opf
from paper_2301_04869_gb300 import synth
from test_gpu_eval_lanes import gpu, hub_network  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limits", [False, True])
def test_same_values_on_both_sides(gpu, limits):  # noqa: F811
    net = hub_network(64, 9, 20)
    if limits:
        net = synth.with_ratings(net, np.ones(net.n_line))
    pd, qd = synth.make_scenarios(net, 381, 0.05, seed=4)
    st = oipm.initial_state(opf.Model(net, pd, qd))
    rng = np.random.default_rng(5)
    st["x"] = st["x"] + 0.005 * rng.standard_normal(st["x"].shape)
    per_scenario = [k for k, v in st.items() if isinstance(v, np.ndarray) and v.ndim == 2]
    want = None
    for N in (379, 380, 381):
        sol = gpu.Solver(net, pd[:N], qd[:N], precision=gpu.PREC_FP64)
        sol.ipm_set_state(sol.pack_state({k: v[:N] if k in per_scenario else v for k, v in st.items()}))
        sol.ipm_eval_derivatives()
        got = [sol.ipm_get_quantity(q, i)[1 if q == gpu.Q_FGH else 0:]
               for q in (gpu.Q_FGH, gpu.Q_JAC) for i in (0, 200, 378)]
        sol.close()
        want = want or got
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a, b)
