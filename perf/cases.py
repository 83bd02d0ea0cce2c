"""Performance cases of the reduced-space interior-point path.

A case is one call sequence that a user of the library makes on one GPU, through
``paper_2301_04869_gb300.ipm`` (the binding of the C ABI):

* ``iteration``  one interior-point iteration (``ipm_step``) over all scenarios from a state in the
  middle of a solve, the state copied in and out on the device: what ``bench.py`` times;
* ``direction``  the Newton direction by its stages (evaluate, condense, factor, solve and refine), what a
  program that brings its own globalisation calls;
* ``solve``      new loads into an existing context and the whole solve from the cold start;
* ``batch``      the same for several uneven instances at once, through the multi-instance runner;
* ``warm``       the warm-start network's forward pass on a batch of load vectors;
* ``train``      one training step of that network.

Networks are the synthetic ones of ``synth.py`` (15 % of the buses with generators below 5,000 buses, 10 %
from there on, as in its workloads); the network belongs to the case, loads and states come from the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2301_04869_gb300 import ipm, synth

PRECISION = {"fp64": ipm.PREC_FP64, "fp64_tc": ipm.PREC_FP64_TC, "mixed": ipm.PREC_MIXED}
BLOCKS = ("x", "u", "s", "y", "z", "zl_x", "zu_x", "zl_u", "zu_u", "zl_s", "zu_s")
STEPS = ("px", "pu", "ps", "py", "pz")

# whole solves stop where power-system programs usually do (MATPOWER's own interior-point solver: 1e-6); a hundred
# times closer the multipliers of active bounds hang on the last digits of the distances to them
SOLVE_TOL = 1e-6

# uneven instances of the multi-instance runner: buses, generators, scenarios, network seed (those of the
# runner's tests, the 1,000-bus one left to the other cases)
UNEVEN = ((30, 6, 1, 0), (60, 9, 5, 0), (100, 15, 8, 3), (150, 22, 12, 5), (200, 30, 3, 7), (120, 18, 17, 9))


def listed():
    def opf(name, kind, n_bus, n_scen, path, rated=False, trips=False, graphs=False):
        return {"name": name, "kind": kind, "n_bus": n_bus, "n_scen": n_scen, "path": path, "rated": rated,
                "trips": trips, "graphs": graphs}
    return [
        # the smallest workload of the benchmark: one scenario of 30 buses, bound by launches and latency
        opf("iteration_30_n1_fp64", "iteration", 30, 1, "fp64"),
        # a network of odd size with line-flow limits and line trips, a few scenarios: everyday contingency study
        opf("direction_119_n7_limits", "direction", 119, 7, "fp64_tc", rated=True, trips=True),
        # a mid-size network and a ragged scenario count on the default path
        opf("direction_433_n19_fp64", "direction", 433, 19, "fp64"),
        # the 1,000-bus workload of the benchmark as the benchmark runs it: replayed graphs, tuned launches
        opf("iteration_1000_n64_fp64_tc", "iteration", 1000, 64, "fp64_tc", graphs=True),
        # the same on the FP64 units and in mixed precision (forward, transposed and multi-vector solves, CG)
        opf("direction_1000_n64_fp64", "direction", 1000, 64, "fp64"),
        opf("direction_1000_n64_mixed", "direction", 1000, 64, "mixed"),
        # between the two benchmark networks: the trailing block no longer fits one multiprocessor
        opf("iteration_3000_n10_fp64_tc", "iteration", 3000, 10, "fp64_tc"),
        # the 10,000-bus network of the headline workload, with as many scenarios as leave room for three contexts
        opf("iteration_10000_n32_mixed", "iteration", 10000, 32, "mixed"),
        # a whole solve of a small network with new loads (rolling re-dispatch)
        opf("solve_120_n17_fp64", "solve", 120, 17, "fp64"),
        # many independent instances of uneven sizes on worker threads
        {"name": "batch_uneven_6", "kind": "batch", "instances": 6, "path": "fp64"},
        # starting points for 1,024 draws of the 1,000-bus network
        {"name": "warm_forward_1024", "kind": "warm", "d_in": 2000, "d_hidden": 512, "d_out": 7395, "rows": 1024},
        # one minibatch of the training of a 120-bus network's warm start
        {"name": "train_120_b256", "kind": "train", "d_in": 240, "d_hidden": 256, "d_out": 893, "rows": 256},
    ]


def draw(rng):
    kind = rng.choice(("iteration", "iteration", "direction", "direction", "direction", "solve", "batch", "warm",
                       "train"))
    path = rng.choice(("fp64", "fp64_tc", "mixed"))
    if kind in ("iteration", "direction"):
        n_bus = int(round(math.exp(rng.uniform(math.log(30), math.log(10000)))))
        # no more scenarios than leave the case below the largest listed one (the FP64 units take about
        # ten times as long as the mixed path on the large networks)
        most = max(1, min(64, int(64 * (1000 / n_bus) ** (1.5 if path == "mixed" else 2.5))))
        n_scen = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
        return {"kind": kind, "n_bus": n_bus, "n_scen": n_scen, "path": path,
                "rated": n_bus <= 1000 and rng.random() < 0.3, "trips": n_bus <= 1000 and rng.random() < 0.3,
                "graphs": kind == "iteration" and n_bus <= 1000 and rng.random() < 0.5}
    if kind == "solve":
        return {"kind": kind, "n_bus": 120, "n_scen": rng.randint(1, 24), "path": rng.choice(("fp64", "fp64_tc")),
                "rated": False, "trips": False, "graphs": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": kind, "instances": rng.randint(2, len(UNEVEN)), "path": "fp64"}
    n_bus = int(round(math.exp(rng.uniform(math.log(30), math.log(1000)))))
    n_gen = max(2, round(0.15 * n_bus))
    n_x, n_u, m = 2 * n_bus - 1 - n_gen, 2 * n_gen - 1, n_gen + 1
    d_out = n_x + n_u + m + 2 * (n_bus - n_gen) + 2 * n_u + 2 * m
    rows = 32 * rng.randint(1, 8) if kind == "train" else int(round(math.exp(rng.uniform(0.0, math.log(1024)))))
    if kind == "train":
        n_bus, d_out = min(n_bus, 250), min(d_out, 1850)
    return {"kind": kind, "d_in": 2 * n_bus, "d_hidden": 128 * rng.randint(1, 4), "d_out": d_out, "rows": rows}


# -- inputs ------------------------------------------------------------------------------------------------


def generators(n_bus):
    return max(2, int(0.15 * n_bus + 0.5) if n_bus < 5000 else int(0.1 * n_bus + 0.5))


def problem(case, seed):
    """(network, pd, qd, tripped lines or None): the case's network, the seed's loads."""
    n_bus, n_scen = case["n_bus"], case["n_scen"]
    net_seed = 9 if case["kind"] == "solve" else 0
    net = synth.make_network(n_bus, generators(n_bus), seed=net_seed, load_scale=0.2 if n_bus >= 5000 else 0.3)
    if case["rated"]:
        net = synth.with_ratings(net, np.random.default_rng(n_bus).uniform(0.8, 2.5, net.n_line))
    pd, qd = synth.make_scenarios(net, n_scen, 0.05, seed=1000 + seed)
    trip = synth.make_contingencies(net, n_scen, seed=2000 + seed) if case["trips"] else None
    return net, pd, qd, trip


def boxes(net):
    """Bounds (lower, upper) of x, u and s in the order of the state vector."""
    n, ng = net.n_bus, net.n_gen
    pq = np.setdiff1d(np.arange(n), net.gen_bus)
    inf = np.full(n - 1, np.inf)
    h_lo, h_up = np.append(-net.qmax, 0.0), np.append(net.qmax, net.pmax[0])
    if net.rate is not None:
        h_lo = np.append(h_lo, np.full(2 * net.n_line, -np.inf))
        h_up = np.append(h_up, np.tile(net.rate ** 2, 2))
    return {"x": (np.append(-inf, net.vmin[pq]), np.append(inf, net.vmax[pq])),
            "u": (np.append(net.vmin[net.gen_bus], np.zeros(ng - 1)), np.append(net.vmax[net.gen_bus], net.pmax[1:])),
            "s": (-h_up, -h_lo)}


def interior_state(net, n_scen, seed):
    """A primal-dual point as the method passes through it in its first ten iterations: inside the boxes,
    complementarity products around ten times the barrier parameter (the method centres by 0.1), angles, voltages
    and prices (from the cost at the slack bus) that differ between neighbours in proportion to the line between
    them (flows around 0.1 pu)."""
    rng = np.random.default_rng([seed, net.n_bus, n_scen])
    n, ng, N = net.n_bus, net.n_gen, n_scen
    box = boxes(net)
    m = box["s"][0].size
    pq = np.setdiff1d(np.arange(n), net.gen_bus)
    z_line = np.hypot(net.r, net.x)

    def along_tree(root, scale, count):  # the first n - 1 lines lead from a bus's parent to the bus
        v = np.full((count, n), float(root))
        noise = scale * z_line[:n - 1] * rng.standard_normal((count, n - 1))
        for line in range(n - 1):
            v[:, net.to[line]] = v[:, net.fr[line]] + noise[:, line]
        return v
    mu = 10.0 ** rng.uniform(-2.2, -1.6)
    volt = np.clip(along_tree(1.0, 0.1, 1), 0.93, 1.07)
    st = {"x": np.concatenate([along_tree(0.0, 0.1, N)[:, 1:],
                               np.clip(volt[:, pq] + 0.002 * rng.standard_normal((N, n - ng)), 0.92, 1.08)], axis=1),
          "u": np.append(volt[0, net.gen_bus], net.pmax[1:] * rng.uniform(0.2, 0.6, ng - 1))}
    lo, up = box["s"]
    up = np.where(np.isfinite(up), up, 0.0)
    st["s"] = lo + (up - lo) * rng.uniform(0.3, 0.7, (N, m))
    st["y"] = np.concatenate([along_tree(net.c1[0], 0.3, N)[:, 1:], along_tree(0.1, 0.3, N)[:, pq]], axis=1) / N
    for k in ("x", "u", "s"):
        lo, up = box[k]
        for side, dist in (("zl_", st[k] - lo), ("zu_", up - st[k])):
            z = 10.0 * mu / dist * rng.uniform(0.5, 1.5, dist.shape)
            st[side + k] = np.where(np.isfinite(dist), z, 0.0)
    st["z"] = st["zl_s"] - st["zu_s"]
    st.update(mu=mu, rho=1.0, delta_last=0.0)
    return st


def mlp_weights(case, seed):
    """(mean, std of the inputs and the outputs), weights in the layout W1, b1, W2, b2, W3, b3."""
    rng = np.random.default_rng([seed, case["d_in"], case["d_hidden"], case["d_out"]])
    d, h, o = case["d_in"], case["d_hidden"], case["d_out"]
    w = [rng.uniform(-1, 1, (h, d)) * math.sqrt(6 / d), 0.05 * rng.standard_normal(h),
         rng.uniform(-1, 1, (h, h)) * math.sqrt(6 / h), 0.05 * rng.standard_normal(h),
         rng.uniform(-1, 1, (o, h)) * math.sqrt(6 / h), 0.05 * rng.standard_normal(o)]
    norm = (rng.uniform(0.1, 0.2, d), rng.uniform(0.02, 0.04, d), rng.standard_normal(o), rng.uniform(0.05, 0.5, o))
    x = norm[0] + norm[1] * rng.standard_normal((case["rows"], d))
    t = norm[2] + norm[3] * rng.standard_normal((case["rows"], o))
    return [a.astype(np.float32) for a in norm], [a.astype(np.float32) for a in w], x.astype(np.float32), t.astype(np.float32)


class State:
    pass


def context(case, seed, st):
    net, pd, qd, trip = problem(case, seed)
    sol = ipm.Solver(net, pd, qd, precision=PRECISION[case["path"]], graphs=case["graphs"], autotune=case["graphs"],
                     tol=SOLVE_TOL if case["kind"] == "solve" else 1e-8)
    if trip is not None:
        sol.ipm_set_contingencies(trip, stream=st.stream)
    return net, pd, qd, sol


def prepare(case, seed):
    st = State()
    st.kind = case["kind"]
    if st.kind in ("warm", "train"):
        norm, w, x, t = mlp_weights(case, seed)
        st.mlp = ipm.MLP(case["d_in"], case["d_hidden"], case["d_out"], max_batch=case["rows"])
        st.mlp.set_params(np.concatenate([a.ravel() for a in w]))
        st.mlp.set_normalization(*norm)
        st.x, st.t = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        return st
    if st.kind == "batch":
        st.members = []
        for i, (n_bus, n_gen, n_scen, net_seed) in enumerate(UNEVEN[:case["instances"]]):
            net, _, _ = synth.screened_network(n_bus, n_gen, n_scen, 0.05, seed=net_seed, scen_seed=1)
            pd, qd = synth.make_scenarios(net, n_scen, 0.02, seed=1000 * i + seed)
            sol = ipm.Solver(net, pd, qd, precision=PRECISION[case["path"]], tol=SOLVE_TOL)
            out = torch.empty(sol.dims.state_len, dtype=torch.float64, device="cuda")
            st.members.append((sol, pd, qd, out))
        return st
    # graphs are replayed on a stream of the program's own (the legacy default stream cannot be captured)
    st.stream = torch.cuda.Stream() if case["graphs"] else torch.cuda.current_stream()
    st.net, st.pd, st.qd, st.sol = context(case, seed, st)
    st.out = torch.empty(st.sol.dims.step_len if st.kind == "direction" else st.sol.dims.state_len,
                         dtype=torch.float64, device="cuda")
    if st.kind != "solve":
        st.at = torch.from_numpy(st.sol.pack_state(interior_state(st.net, case["n_scen"], seed))).cuda()
    st.stream.wait_stream(torch.cuda.current_stream())
    return st


def run(st):
    if st.kind == "warm":
        return st.mlp.forward(st.x)
    if st.kind == "train":
        loss = st.mlp.train_step(st.x, st.t, 1e-3)
        return {"loss": loss, "params": st.mlp.get_params()}
    if st.kind == "batch":
        for sol, pd, qd, _ in st.members:
            sol.ipm_set_loads(pd, qd)
        torch.cuda.current_stream().synchronize()  # the runner works on streams of its own
        _, _, status, _ = ipm.ipm_solve_batch([m[0] for m in st.members])
        assert not status.any(), status
        return [m[0].ipm_get_state(m[3]) for m in st.members]
    sol, stream = st.sol, st.stream
    if st.kind == "solve":
        sol.ipm_set_loads(st.pd, st.qd, stream=stream)
        sol.ipm_solve(stream=stream)
        sol.ipm_get_state(st.out, stream=stream)
    elif st.kind == "iteration":
        sol.ipm_set_state(st.at, stream=stream)
        sol.ipm_step(stream=stream)
        sol.ipm_get_state(st.out, stream=stream)
    else:
        sol.ipm_set_state(st.at, stream=stream)
        sol.ipm_eval_derivatives(stream=stream)
        sol.ipm_condense_scenarios(stream=stream)
        delta = 0.0
        while not sol.ipm_factor_schur(delta, stream=stream):
            delta = 100.0 * delta or 1e-4
        sol.ipm_solve_kkt(st.out, stream=stream)
    torch.cuda.current_stream().wait_stream(stream)
    return steps(sol, st.out) if st.kind == "direction" else blocks(sol, st.out)


def blocks(sol, v):
    return {k: b for k, b in sol.split_state(v).items() if k in BLOCKS}


def steps(sol, v):
    return sol.split_step(v)


# -- what a pass cannot do without -------------------------------------------------------------------------


def opf_work(case, iterations):
    """Inputs, outputs and multiply-adds of the reduction: with N scenarios, n_x states and n_u controls the
    dense product Z^T Y (symmetric, n_x n_u^2 multiply-adds), the solves with the factors of G_x for the n_u
    columns and the Cholesky of K_hat.  The factors have about 20 entries a state on the smaller networks."""
    n, N = case["n_bus"], case["n_scen"]
    ng = generators(n)
    n_x, n_u, m = 2 * n - 1 - ng, 2 * ng - 1, ng + 1 + (2 * int(1.35 * n + 0.5) if case["rated"] else 0)
    lu = 20 * n_x + (0.09 * n_x) ** 2
    state = 8 * (4 * N * n_x + 4 * N * m + 3 * n_u)
    flops = N * (n_x * n_u * n_u + 2 * lu * n_u + 2 * (0.09 * n_x) ** 3 / 3) + n_u ** 3 / 3
    return {"bytes": iterations * 2 * state, "flops": iterations * flops}


def work(case):
    if case["kind"] in ("warm", "train"):
        d, h, o, b = case["d_in"], case["d_hidden"], case["d_out"], case["rows"]
        w = d * h + h * h + o * h
        if case["kind"] == "warm":
            return {"bytes": 4 * (b * (d + o) + w), "flops": 2 * b * w}
        return {"bytes": 4 * (b * (d + o) + 6 * w), "flops": 6 * b * w}
    if case["kind"] == "batch":
        parts = [opf_work({"n_bus": n, "n_scen": N, "rated": False}, 20) for n, _, N, _ in UNEVEN[:case["instances"]]]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return opf_work(case, 20 if case["kind"] == "solve" else 1)


# -- the same in 64 bits, by dense algebra -----------------------------------------------------------------


class Model:
    """The power-flow functions of the cases by line ends, for automatic differentiation: bus angles and
    magnitudes from (x, u), balances g, limited quantities h, cost f."""

    def __init__(self, net, n_scen):
        dev = self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a, k=torch.float64: torch.as_tensor(np.asarray(a), dtype=k, device=dev)  # noqa: E731
        self.net, self.N = net, n_scen
        n, ng = net.n_bus, net.n_gen
        pq = np.setdiff1d(np.arange(n), net.gen_bus)
        y = 1.0 / (net.r + 1j * net.x)
        self.ends = [(t(a, torch.long), t(b, torch.long)) for a, b in ((net.fr, net.to), (net.to, net.fr))]
        self.gs, self.bs, self.bh = t(y.real), t(y.imag), t(net.b / 2)
        self.n, self.ng, self.pq, self.gen = n, ng, t(pq, torch.long), t(net.gen_bus, torch.long)
        vpos = np.empty(n, dtype=np.int64)  # where a bus's magnitude sits in (x, u)
        vpos[pq], vpos[net.gen_bus] = n - 1 + np.arange(pq.size), 2 * n - 1 - ng + np.arange(ng)
        self.vpos, self.n_x, self.n_u = t(vpos, torch.long), 2 * n - 1 - ng, 2 * ng - 1
        # bus sums of line-end quantities, from ends then to ends
        S = torch.zeros((n, 2 * net.n_line), dtype=torch.float64, device=dev)
        S[torch.cat([e[0] for e in self.ends]), torch.arange(2 * net.n_line, device=dev)] = 1.0
        self.sum = S
        self.c2, self.c1 = t(net.c2), t(net.c1)
        self.box = {k: (t(lo), t(up)) for k, (lo, up) in boxes(net).items()}
        self.m = self.box["s"][0].numel()

    def functions(self, w, pd, qd, on):
        """(f, g, h) at w = (x, u) of one scenario."""
        n, ng = self.n, self.ng
        theta = torch.cat([torch.zeros_like(w[:1]), w[:n - 1]])
        v = w[self.vpos]
        pg = w[self.n_x + ng:]
        P, Q = [], []
        for a, b in self.ends:
            d = theta[a] - theta[b]
            va, vb = v[a], v[b]
            c, s = torch.cos(d), torch.sin(d)
            P.append(on * (va * va * self.gs - va * vb * (self.gs * c + self.bs * s)))
            Q.append(on * (-va * va * (self.bs + self.bh) - va * vb * (self.gs * s - self.bs * c)))
        P, Q = torch.cat(P), torch.cat(Q)
        bus_p, bus_q = self.sum @ P + pd, self.sum @ Q + qd
        inj = torch.zeros_like(bus_p).index_add(0, self.gen[1:], pg)
        slack = bus_p[0]
        g = torch.cat([(bus_p - inj)[1:], bus_q[self.pq]])
        h = torch.cat([bus_q[self.gen], slack[None]])
        if self.net.rate is not None:
            h = torch.cat([h, P * P + Q * Q])
        f = (self.c2[0] * slack * slack + self.c1[0] * slack + (self.c2[1:] * pg * pg + self.c1[1:] * pg).sum()) / self.N
        return f, g, h


def exact_direction(M, st, loads, mu):
    """Newton step of the barrier problem at `st` (tensors), by dense algebra per scenario; also the pieces that
    the rules of an iteration read: objective gradients, residuals, K p."""
    n_x, n_u, N = M.n_x, M.n_u, M.N
    inv = lambda d: torch.where(torch.isfinite(d), 1.0 / d, torch.zeros_like(d))  # noqa: E731
    sig, bar = {}, {}
    for k in ("x", "u", "s"):
        lo, up = M.box[k]
        il, iu = inv(st[k] - lo), inv(up - st[k])
        sig[k] = st["zl_" + k] * il + st["zu_" + k] * iu
        bar[k] = mu * (iu - il)  # gradient of the barrier terms
    eye = torch.eye(n_x + n_u, dtype=torch.float64, device=M.dev)
    K_hat = torch.diag(sig["u"])
    rhs = -bar["u"].clone()
    keep = []
    for i in range(N):
        w = torch.cat([st["x"][i], st["u"]])
        y, z = st["y"][i], st["z"][i]
        fun = lambda w: M.functions(w, *loads[i])  # noqa: E731,B023
        gh = lambda w: torch.cat(fun(w)[1:])  # noqa: E731,B023
        lag = lambda w: (lambda f, g, h: f + y @ g + z @ h)(*fun(w))  # noqa: E731,B023
        pull = torch.func.vjp(gh, w)[1]
        rows = torch.eye(n_x + M.m, dtype=torch.float64, device=M.dev)
        JH = torch.cat([torch.func.vmap(lambda r: pull(r)[0])(c) for c in rows.split(1024)])  # noqa: B023
        grad = torch.func.grad(lag)
        W = torch.cat([torch.func.vmap(lambda d: torch.func.jvp(grad, (w,), (d,))[1])(c) for c in eye.split(1024)])  # noqa: B023
        gf = torch.func.grad(lambda w: fun(w)[0])(w)
        f, g, h = fun(w)
        G, H = JH[:n_x], JH[n_x:]
        r4 = h + st["s"][i]
        r2 = z + bar["s"][i]  # gradient of the barrier Lagrangian in s
        r1 = gf + G.T @ y + H.T @ z
        r1[:n_x] += bar["x"][i]
        Ss = sig["s"][i]
        K = W + H.T @ (Ss[:, None] * H)
        K[:n_x, :n_x] += torch.diag(sig["x"][i])
        rh = r1 + H.T @ (Ss * r4 - r2)
        LU = torch.linalg.lu_factor(G[:, :n_x])
        sol = -torch.linalg.lu_solve(*LU, torch.cat([G[:, n_x:], g[:, None]], 1))
        Z, b = sol[:, :n_u], sol[:, n_u]
        T = torch.cat([Z, torch.eye(n_u, dtype=torch.float64, device=M.dev)])
        K_hat = K_hat + T.T @ (K @ T)
        rhs = rhs - T.T @ (rh + K[:, :n_x] @ b)
        keep.append((w, G, H, K, W, LU, Z, b, rh, r2, r4, gf, f, g, h))
    C, bad = torch.linalg.cholesky_ex(K_hat)
    if int(bad):
        return None
    pu = torch.cholesky_solve(rhs[:, None], C)[:, 0]
    p = {k: [] for k in STEPS}
    for i, (w, G, H, K, W, LU, Z, b, rh, r2, r4, *_) in enumerate(keep):
        px = Z @ pu + b
        pw = torch.cat([px, pu])
        py = -torch.linalg.lu_solve(*LU, (rh + K @ pw)[:n_x, None], adjoint=True)[:, 0]
        ps = -r4 - H @ pw
        pz = -r2 - sig["s"][i] * ps
        for k, v in zip(STEPS, (px, None, ps, py, pz)):
            p[k].append(v)
    p = {k: pu if k == "pu" else torch.stack(v) for k, v in p.items()}
    return p, keep, sig, bar


def exact_iteration(M, st, loads):
    """One iteration of the method from `st`: centring from the mean complementarity, fraction to the boundary,
    backtracking on the l1 merit, safeguarded bound duals."""
    N, n_x = M.N, M.n_x
    finite = {(k, side): torch.isfinite(b).expand_as(st[k]) for k in ("x", "u", "s") for side, b in zip("lu", M.box[k])}

    def gaps(v):
        return {(k, side): torch.where(finite[k, side], (v[k] - b) if side == "l" else (b - v[k]), 1.0)
                for k in ("x", "u", "s") for side, b in zip("lu", M.box[k])}
    d0 = gaps(st)
    dual = {(k, side): st["z%s_%s" % (side, k)] for k, side in d0}
    total = sum((dual[q] * d0[q])[finite[q]].sum() for q in d0)
    mu = max(1e-9, 0.1 * float(total / sum(int(finite[q].sum()) for q in d0)))
    found = exact_direction(M, st, loads, mu)
    if found is None:
        return None
    p, keep, sig, bar = found
    pw = {"x": p["px"], "u": p["pu"], "s": p["ps"]}
    sign = {"l": 1.0, "u": -1.0}
    dz = {q: torch.where(finite[q], mu / d0[q] - dual[q] - sign[q[1]] * dual[q] / d0[q] * pw[q[0]], 0.0) for q in d0}
    tau = max(0.99, 1.0 - mu)

    def longest(room, d):
        return min(1.0, float(torch.where(d < 0, -tau * room / d, torch.inf).min()))
    a_max = min(longest(d0[q][finite[q]], sign[q[1]] * pw[q[0]][finite[q]]) for q in d0 if finite[q].any())
    a_dual = min(longest(dual[q][finite[q]], dz[q][finite[q]]) for q in d0 if finite[q].any())
    slope = float(p["pu"] @ bar["u"] + (p["px"] * bar["x"]).sum() + (p["ps"] * bar["s"]).sum())
    curv = float(p["pu"] @ (sig["u"] * p["pu"]) + (sig["s"] * p["ps"] ** 2).sum() + (sig["x"] * p["px"] ** 2).sum())
    c1 = 0.0
    for i, (w, G, H, K, W, LU, Z, b, rh, r2, r4, gf, f, g, h) in enumerate(keep):
        v = torch.cat([p["px"][i], p["pu"]])
        slope += float(gf @ v)
        curv += float(v @ (W @ v))
        c1 += float(g.abs().sum() + r4.abs().sum())
    rho = st["rho"]
    if c1 > 0.0:
        rho = max(rho, (slope + 0.5 * max(curv, 0.0)) / (0.9 * c1))

    def merit(v):
        phi, off = 0.0, 0.0
        for i in range(N):
            f, g, h = M.functions(torch.cat([v["x"][i], v["u"]]), *loads[i])
            phi, off = phi + float(f), off + float(g.abs().sum() + (h + v["s"][i]).abs().sum())
        gap = gaps(v)
        return phi - mu * sum(float(torch.log(gap[q][finite[q]]).sum()) for q in gap) + rho * off
    phi0 = merit(st)
    alpha = a_max
    while True:
        new = {k: st[k] + alpha * pw[k] for k in ("x", "u", "s")}
        if merit(new) - phi0 <= 1e-4 * alpha * (slope - rho * c1) + 10 * np.finfo(float).eps * abs(phi0):
            break
        alpha *= 0.5
        if alpha < 1e-12:
            return None
    new["y"], new["z"] = st["y"] + alpha * p["py"], st["z"] + alpha * p["pz"]
    for q, gap in gaps(new).items():
        z = torch.minimum(torch.maximum(dual[q] + a_dual * dz[q], mu / (1e10 * gap)), 1e10 * mu / gap)
        new["z%s_%s" % (q[1], q[0])] = torch.where(finite[q], z, 0.0)
    return {k: new[k] for k in BLOCKS}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("warm", "train"):
        norm, w, x, t = mlp_weights(case, seed)
        im, istd, om, ostd = (torch.from_numpy(a).double() for a in norm)
        W1, b1, W2, b2, W3, b3 = (torch.from_numpy(a).double() for a in w)
        gelu = torch.nn.functional.gelu
        out = gelu(gelu((torch.from_numpy(x).double() - im) / istd @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
        if kind == "warm":
            return om + ostd * out
        # the weights after a step of Adam hang on the signs of gradients near zero: no value in 64 bits
        return None
    if kind in ("solve", "batch") or case["n_bus"] > 1000 or case["n_bus"] ** 2 * case["n_scen"] > 7e7:
        return None  # a whole solve, or dense algebra that takes too long
    net, pd, qd, trip = problem(case, seed)
    M = Model(net, case["n_scen"])
    st = {k: torch.as_tensor(v, device=M.dev) if isinstance(v, np.ndarray) else v
          for k, v in interior_state(net, case["n_scen"], seed).items()}
    loads = []
    for i in range(case["n_scen"]):
        on = np.ones(net.n_line)
        if trip is not None and trip[i] >= 0:
            on[trip[i]] = 0.0
        loads.append(tuple(torch.as_tensor(a, device=M.dev) for a in (pd[i], qd[i], on)))
    if kind == "iteration":
        return exact_iteration(M, st, loads)
    found = exact_direction(M, st, loads, st["mu"])
    return found and found[0]


if __name__ == "__main__":
    for c in listed() + [draw(random.Random(i)) for i in range(12)]:
        print(c, work(c))
