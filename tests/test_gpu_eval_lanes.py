"""The model functions and their derivatives on both sides of the size at which
a (bus, scenario) pair goes from eight lanes to one (38,912 pairs), on the
smallest network, and with a bus of more than 20 incident lines (three for some
lanes): g, h, the Jacobians and the condensed Hessian blocks of the first and
the last scenario against the oracle at 1e-10, with and without line limits."""
import dataclasses

import numpy as np
import pytest

from oracle import ipm as oipm
from oracle import kkt, opf
from paper_2301_04869_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-10


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


def hub_network(n, ng, extra):
    """A synthetic network with `extra` more lines from bus n - 1 (with the
    first lines' constants)."""
    net = synth.make_network(n, ng, seed=2)
    near = np.r_[net.to[net.fr == n - 1], net.fr[net.to == n - 1], n - 1]
    to = np.setdiff1d(np.arange(n), near)[:extra].astype(net.to.dtype)
    return dataclasses.replace(
        net, fr=np.r_[net.fr, np.full(extra, n - 1, net.fr.dtype)], to=np.r_[net.to, to],
        **{k: np.r_[getattr(net, k), getattr(net, k)[:extra]] for k in ("r", "x", "b")})


@pytest.mark.parametrize("n,ng,N,extra,limits", [
    (5, 2, 1, 0, False), (41, 6, 1, 20, False), (41, 6, 3, 20, True),
    (64, 9, 607, 20, True), (64, 9, 608, 20, True), (64, 9, 609, 0, False)])
def test_functions_and_derivatives(gpu, n, ng, N, extra, limits):
    net = hub_network(n, ng, extra)
    if limits:
        net = synth.with_ratings(net, np.ones(net.n_line))
    pd, qd = synth.make_scenarios(net, N, 0.05, seed=4)
    M = opf.Model(net, pd, qd)
    st = oipm.initial_state(M)
    rng = np.random.default_rng(5)
    st["x"] = st["x"] + 0.005 * rng.standard_normal(st["x"].shape)
    st["z"] = rng.standard_normal(st["z"].shape)
    st["y"] = rng.standard_normal(st["y"].shape)
    Sx, _, Ss = kkt.sigmas(M, st)
    sol = gpu.Solver(net, pd, qd, precision=gpu.PREC_FP64)
    nx, nu, m = sol.dims.n_x, sol.dims.n_u, sol.dims.m
    sol.ipm_set_state(sol.pack_state(st))
    sol.ipm_eval_derivatives()
    sol.ipm_condense_scenarios()
    for i in sorted({0, N - 1}):
        o = M.derivatives(i, st["x"][i], st["u"], st["y"][i], st["z"][i])
        assert rel(sol.ipm_get_quantity(gpu.Q_FGH, i)[1:1 + nx], o["g"]) <= TOL
        assert rel(sol.ipm_get_quantity(gpu.Q_FGH, i)[1 + nx:], o["h"]) <= TOL
        jac = sol.ipm_get_quantity(gpu.Q_JAC, i)
        got = np.split(jac, np.cumsum([nx * nx, nx * nu, m * nx]))
        for a, k, r in zip(got, ("Gx", "Gu", "Hx", "Hu"), (nx, nx, m, m)):
            assert rel(a.reshape(r, -1), o[k].toarray()) <= TOL
        got = np.split(sol.ipm_get_quantity(gpu.Q_HESS, i), np.cumsum([nx * nx, nx * nu]))
        want = kkt.condensed_blocks(o, Sx[i], Ss[i], np.zeros(nx), np.zeros(m), np.zeros(m), 0.0)
        for a, b in zip(got, want[:3]):
            assert rel(a.reshape(b.shape), b.toarray()) <= TOL
    sol.close()
