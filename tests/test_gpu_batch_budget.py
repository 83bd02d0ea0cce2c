"""Admission of the multi-instance runner under a device memory budget: two
instances whose contexts do not fit the budget together (the solve's panels
counted: of 310 MB of a 1,000-bus context with 16 scenarios they take 77) run
one after the other."""
import pytest

from paper_2301_04869_gb300 import synth

pytestmark = pytest.mark.gpu


def test_two_contexts_past_the_budget_run_in_turn():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2301_04869_gb300 import ipm
    net = synth.make_network(1000, 150, seed=0, load_scale=0.3)
    pd, qd = synth.make_scenarios(net, 16, 0.02, seed=1)
    ipm.Solver(net, pd, qd).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sol = ipm.Solver(net, pd, qd)
    size = free - torch.cuda.mem_get_info()[0]
    sol.close()
    budget = 560 << 20
    assert size < budget < 2 * size
    _, _, status, stats, _ = ipm.ipm_run_instances([net, net], [pd, pd], [qd, qd], mem_budget=budget, tol=1e-3,
                                                   n_threads=2)
    assert not status.any()
    assert stats["max_active"] == 1
