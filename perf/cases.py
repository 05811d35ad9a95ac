"""The work a user of this framework has it do, as cases that can be timed.

Every case goes through the public entry points of ``paper_2410_17203_gb300``
as a user's program calls them: cold solves of one instance (``opf_reset``,
``opf_iterate``, ``opf_solution``) from the smallest named workload to the
largest, at even, odd and long horizons and over-relaxed; a re-solve from a
previous state; a batch of instances; the unrolled cost and its gradients; and
the training gradient of the warm-start network.  Instances come from
``gridgen`` (the named workloads and the same recipe at other sizes); a seed
draws other loads (and features, targets, weights) for the same network.

``exact`` restates each path in plain FP64 PyTorch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from gridgen import make_case, scale_case

F64 = torch.float64

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def _solve(name, n_nodes, T, K, iters, config="", alpha=1.0, n_hvdc=0):
    return dict(name=name, kind="solve", config=config, n_nodes=n_nodes, T=T, K=K, iters=iters, alpha=alpha,
                n_hvdc=n_hvdc)


def listed():
    return [
        # the smallest workload (30 buses, one period, five outages): a solve is all launch latency
        _solve("solve-tiny", 30, 1, 5, 100, config="tiny"),
        # a small grid over an odd horizon with HVDC links: scalar accesses, ragged rows
        _solve("solve-301-odd", 301, 31, 7, 100, n_hvdc=3),
        # a day of a 2,000-bus system with 20 outages: the ordinary single solve
        _solve("solve-2k", 2000, 24, 20, 100, config="2k"),
        # a single period of a 5,000-bus system (security-constrained dispatch of the next hour)
        _solve("solve-5k-1t", 5000, 1, 20, 100),
        # a week of hours: beyond the horizons the inner ADMM keeps in registers
        _solve("solve-week", 500, 168, 4, 50),
        # the headline workload: 10,000 buses, four days, 50 outages
        _solve("solve-10k", 10000, 96, 50, 50, config="10k"),
        # over-relaxed message passing, two days of 1,000 buses
        _solve("solve-relaxed", 1000, 48, 20, 100, alpha=1.5),
        # a re-solve of the 2,000-bus day after its loads moved, from the previous
        # state and penalties kept on the device, and the new state back
        dict(name="resolve-2k", kind="resolve", config="2k", n_nodes=2000, T=24, K=20, iters=96),
        # planning: independent instances of mixed sizes and horizons as one batch
        dict(name="batch-16", kind="batch", n_inst=16, first=1000, n_max=3000, iters=50),
        # cost and gradients through unrolled iterations, the ordinary size
        dict(name="grad-2k", kind="grad", config="2k", n_nodes=2000, T=24, K=20, iters=50),
        # the same on a small grid with an odd horizon, more iterations
        dict(name="grad-151-odd", kind="grad", config="", n_nodes=151, T=31, K=3, iters=60),
        # one training gradient of the warm-start network on the 2,000-bus day
        dict(name="net-2k", kind="net", config="2k", n_nodes=2000, T=24, K=20, F=9),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["resolve", "batch", "grad", "grad", "net"])
    if kind == "batch":
        return dict(kind="batch", n_inst=rng.randint(3, 16), first=rng.randint(2000, 99000),
                    n_max=_log_uniform(rng, 300, 3000), iters=10 * rng.randint(2, 5))
    if kind == "net":
        n = _log_uniform(rng, 30, 2000)
        return dict(kind="net", config="", n_nodes=n, T=rng.randint(1, 24), K=0, F=rng.choice([6, 9, 9, 16]))
    T = rng.choice([1, 3, 7, 12, 24, 24, 31, 48, 48, 96, 100, 168])
    if kind == "grad":
        T = rng.choice([1, 6, 7, 12, 24, 31, 48])
        n = _log_uniform(rng, 30, 2000)
        K = _log_uniform(rng, 1, 21) - 1
        while (K + 1) * n * T > 21 * 2000 * 24:
            n = max(30, n // 2)
        return dict(kind="grad", config="", n_nodes=n, T=T, K=K, iters=rng.randint(20, 60))
    n = _log_uniform(rng, 30, 10000)
    K = _log_uniform(rng, 1, 51) - 1
    while (K + 1) * n * T > 12_000_000:
        n = max(30, n // 2)
    if kind == "resolve":
        while (K + 1) * n * T > 2_000_000:
            n = max(30, n // 2)
        return dict(kind="resolve", config="", n_nodes=n, T=T, K=K, iters=10 * rng.randint(2, 9) + 6)
    alpha = rng.choice([1.0, 1.0, 1.0, 1.0, 1.5, 1.7])
    iters = rng.randint(20, 50) if (K + 1) * n * T > 2_000_000 else rng.randint(40, 100)
    c = _solve("", n, T, K, iters, alpha=alpha, n_hvdc=rng.choice([0, 0, 2]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


@functools.lru_cache(maxsize=8)
def _network(config, n_nodes, T, K, n_hvdc):
    if config:
        return make_case(config)
    # small grids keep enough non-bridge lines for their outages
    K = min(K, max(0, n_nodes // 5))
    return make_case(scale_case(n_nodes, T, K, seed=n_nodes + T, n_hvdc=n_hvdc))


def _instance(case, seed):
    """The case's network with every load scaled by lognormal(0, 0.15) per step."""
    base = _network(case["config"], case["n_nodes"], case["T"], case["K"], case.get("n_hvdc", 0))
    c = dict(base)
    rng = np.random.default_rng(seed)
    c["load_p"] = base["load_p"] * rng.lognormal(0.0, 0.15, size=base["load_p"].shape)
    return c


def _batch_instances(case, seed):
    """Buses log-uniform in [100, n_max], T in {1, 24, 48}, 0..20 outages."""
    rng = np.random.default_rng(case["first"])
    out = []
    for i in range(case["n_inst"]):
        n = int(round(float(np.exp(rng.uniform(np.log(100), np.log(case["n_max"]))))))
        T, K = int(rng.choice([1, 24, 48])), int(rng.integers(0, 21))
        out.append(_instance(dict(config="", n_nodes=n, T=T, K=K), seed + i))
    return out


PREVIOUS_ITERS = 60   # iterations behind the state a re-solve starts from


@functools.lru_cache(maxsize=2)
def _previous(config, n_nodes, T, K):
    """State (float32, host) and penalties after some iterations on the
    network's own loads, what a user keeps of the previous solve."""
    r = _Iteration(_network(config, n_nodes, T, K, 0))
    for _ in range(PREVIOUS_ITERS):
        r.step()
    st = {k: v.to("cpu", torch.float32) for k, v in r.state().items()}
    return st, r.rho_p, r.rho_th


NET_SCALE = (1.0, 4.0)


def _net_inputs(case, seed):
    """Features and targets [T * N, .] of every (step, node), and the weights
    of a network in training (layer order of include/opf_wsnet.h)."""
    net = _network(case["config"], case["n_nodes"], case["T"], case["K"], 0)
    rng = np.random.default_rng(seed)
    R, F = net["n_nodes"] * net["T"], case["F"]
    X = rng.normal(size=(R, F)).astype(np.float32)
    Y = rng.normal(size=(R, 2)).astype(np.float32)
    parts = []
    for shp in [(F, 64), (64,)] + [(64, 64), (64, 64), (64,)] * 3 + [(64, 2), (2,)]:
        if len(shp) == 2:
            lim = math.sqrt(6.0 / shp[0])
            parts.append(rng.uniform(-lim, lim, size=shp))
        else:
            parts.append(0.05 * rng.normal(size=shp))
    flat = np.concatenate([p.ravel() for p in parts]).astype(np.float32)
    return net, X, Y, flat


class _Batch:
    """A batch and the solvers it groups."""

    def __init__(self, solvers):
        import paper_2410_17203_gb300 as opf
        self.opf, self.solvers = opf, solvers
        self.h = opf.opf_batch_create([s.h for s in solvers])
        opf.opf_batch_autotune(self.h, steps=10)

    def __del__(self):
        self.opf.opf_batch_destroy(self.h)


def _solution_buffers(info):
    Kp, L, N, S, T = info["k_count"], info["L"], info["N"], info["S"], info["T"]
    z = functools.partial(torch.zeros, dtype=torch.float32, device="cuda")
    return dict(p_dev=z((S, T)), p_line=z((Kp, L, T)), theta_node=z((Kp, N, T)), price=z((N, T)))


def prepare(case, seed):
    import paper_2410_17203_gb300 as opf
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "solve":
        s = opf.Solver(_instance(case, seed), dict(alpha=case["alpha"]), stream=stream)
        return dict(case=case, solver=s, out=_solution_buffers(s.info))
    if kind == "resolve":
        st, rho_p, rho_th = _previous(case["config"], case["n_nodes"], case["T"], case["K"])
        s = opf.Solver(_instance(case, seed), dict(rho_p=rho_p, rho_theta=rho_th), stream=stream)
        return dict(case=case, solver=s, prev={k: v.cuda() for k, v in st.items()},
                    out={k: torch.zeros(shp, dtype=torch.float32, device="cuda")
                         for k, shp in opf.state_shapes(s.info).items()})
    if kind == "batch":
        solvers = [opf.Solver(c, stream=stream) for c in _batch_instances(case, seed)]
        return dict(case=case, batch=_Batch(solvers), outs=[_solution_buffers(s.info) for s in solvers])
    if kind == "grad":
        c = _instance(case, seed)
        d = opf.UnrolledCost(c, rho_p=1.0, rho_theta=1.0, checkpoint_every=20, stream=stream)
        x = {k: torch.as_tensor(np.asarray(c[k], np.float32), device="cuda") for k in ("load_p", "gen_pmax", "line_u")}
        return dict(case=case, diff=d, x=x)
    net, X, Y, flat = _net_inputs(case, seed)
    w = opf.WarmStartNet(net["n_nodes"], net["line_from"], net["line_to"], net["line_b"], net["T"], case["F"],
                         params=flat, stream=stream)
    return dict(case=case, net=w, x=torch.from_numpy(X).cuda(), y=torch.from_numpy(Y).cuda())


def run(state):
    import paper_2410_17203_gb300 as opf
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        s, out = state["solver"], state["out"]
        opf.opf_reset(s.h)
        s.iterate(case["iters"])
        return dict(out, objective=opf.opf_solution(s.h, on_device=True, objective=True, **out))
    if kind == "resolve":
        s, out = state["solver"], state["out"]
        opf.opf_reset(s.h)
        opf.opf_set_state(s.h, state["prev"], on_device=True)
        s.iterate(case["iters"])
        return dict(opf.opf_get_state(s.h, on_device=True, out=out))
    if kind == "batch":
        b = state["batch"]
        for s in b.solvers:
            opf.opf_reset(s.h)
        opf.opf_batch_iterate(b.h, case["iters"])
        for s, out in zip(b.solvers, state["outs"]):
            opf.opf_solution(s.h, on_device=True, objective=False, **out)
        return state["outs"]
    if kind == "grad":
        x = state["x"]
        f, g = state["diff"].cost_grad_device(case["iters"], x["load_p"], x["gen_pmax"], x["line_u"])
        return dict(g, cost=f)
    loss, g = state["net"].gradient(state["x"], state["y"], NET_SCALE)
    return dict(loss=loss, grad=g)


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------


def _iteration_work(net):
    """Bytes and operations of one iteration: every FP32 element of the
    iterate (lines p, theta_1, theta_2, v_1, v_2; nodes u, pbar, theta_bar;
    device powers) read once and written once; about 60 operations per line
    item, 20 per node and contingency, and the inner ADMM's ten iterations of
    about 120 per step of a battery and 60 of a ramp-limited generator."""
    N, L, T, Kp = net["n_nodes"], len(net["line_from"]), net["T"], len(net["outaged"]) + 1
    G, D, B = len(net["gen_node"]), len(net["load_node"]), len(net["stor_node"])
    S = G + D + B + 2 * len(net["hvdc_from"])
    nbytes = 8 * Kp * T * (5 * L + 3 * N) + 8 * S * T
    flops = Kp * T * (60 * L + 20 * N) + 10 * T * (60 * G + 120 * B)
    return nbytes, flops, dict(N=N, L=L, T=T, Kp=Kp, S=S)


def work(case):
    kind = case["kind"]
    if kind == "net":
        net = _network(case["config"], case["n_nodes"], case["T"], case["K"], 0)
        R, F = net["n_nodes"] * net["T"], case["F"]
        C = F * 64 + 64 + 3 * (2 * 64 * 64 + 64) + 128 + 2
        # features, targets and the kept activations (H0..H3 and the neighbour
        # averages, written forward and read backward); products of the
        # forward pass, the input gradients and the weight gradients
        macs = R * (F * 64 + 3 * 2 * 64 * 64 + 128)
        return dict(bytes=4 * R * (F + 4) + 2 * 4 * R * 64 * 7 + 8 * C, flops=2 * 3 * macs)
    if kind == "batch":
        nbytes = flops = 0
        for c in _batch_instances(case, 0):
            b, f, d = _iteration_work(c)
            nbytes += case["iters"] * b + 4 * (d["S"] + d["Kp"] * (d["L"] + d["N"]) + d["N"]) * d["T"]
            flops += case["iters"] * f
        return dict(bytes=nbytes, flops=flops)
    b, f, d = _iteration_work(_network(case["config"], case["n_nodes"], case["T"], case["K"], case.get("n_hvdc", 0)))
    if kind == "grad":
        # forward, and a reverse pass over the adjoint of every state array
        return dict(bytes=2 * case["iters"] * b, flops=3 * case["iters"] * f)
    io = 4 * (d["S"] + d["Kp"] * (d["L"] + d["N"]) + d["N"]) * d["T"]
    if kind == "resolve":
        io = 2 * 4 * (d["S"] + d["Kp"] * (5 * d["L"] + d["N"])) * d["T"]
    return dict(bytes=case["iters"] * b + io, flops=case["iters"] * f)


# ---------------------------------------------------------------------------
# the same in FP64
# ---------------------------------------------------------------------------


def _ramp_rows(T):
    """A of p <= pmax, -p <= -pmin, and the ramp limits of consecutive steps."""
    I = torch.eye(T, dtype=F64)
    D = I[1:] - I[:-1]
    return torch.cat([I, -I, D, -D])


def _battery_rows(T, eff):
    """A over (p, c, delta, s) and its equality rows, in the row order of
    opf_get_info: p + c - delta = 0, the state of charge, s_1 = s_{T+1} = 0,
    then the upper and lower limits of c, delta and s."""
    n = 4 * T + 1
    A = torch.zeros((8 * T + 4, n), dtype=F64)
    t = torch.arange(T)
    A[t, t], A[t, T + t], A[t, 2 * T + t] = 1.0, 1.0, -1.0
    A[T + t, 3 * T + t + 1], A[T + t, 3 * T + t], A[T + t, T + t], A[T + t, 2 * T + t] = 1.0, -1.0, -eff, 1.0
    A[2 * T, 3 * T], A[2 * T + 1, 4 * T] = 1.0, 1.0
    r = 2 * T + 2
    for first, cnt in ((T, T), (2 * T, T), (3 * T, T + 1)):
        i = torch.arange(cnt)
        A[r + i, first + i] = 1.0
        A[r + cnt + i, first + i] = -1.0
        r += 2 * cnt
    eq = torch.zeros(8 * T + 4, dtype=torch.bool)
    eq[:2 * T + 2] = True
    return A, eq


class _Iteration:
    """The message-passing iteration (Sections 3.1 to 3.6, Appendix D) on FP64
    tensors, with explicit copies z, xi of every terminal."""

    def __init__(self, net, alpha=1.0, rho_p=1.0, rho_th=1.0, adapt_every=10, params=None):
        dev = self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")

        def f(a):
            return torch.as_tensor(np.asarray(a), dtype=F64, device=dev)

        def i(a):
            return torch.as_tensor(np.asarray(a), dtype=torch.long, device=dev)

        self.alpha, self.rho_p, self.rho_th, self.adapt_every, self.it = alpha, rho_p, rho_th, adapt_every, 0
        self.T, self.N, self.L = T, N, L = int(net["T"]), int(net["n_nodes"]), len(net["line_from"])
        self.Kp = Kp = len(net["outaged"]) + 1
        self.G, self.D, self.B = len(net["gen_node"]), len(net["load_node"]), len(net["stor_node"])
        self.H = len(net["hvdc_from"])
        hv = np.stack([net["hvdc_from"], net["hvdc_to"]], 1).ravel()
        self.line_node = i(np.concatenate([net["line_from"], net["line_to"]]))
        self.dev_node = i(np.concatenate([net["gen_node"], net["load_node"], net["stor_node"], hv]))
        self.S = len(self.dev_node)
        cth = torch.zeros(N, dtype=F64, device=dev).index_add(0, self.line_node, torch.ones(2 * L, dtype=F64, device=dev))
        cnt = cth.index_add(0, self.dev_node, torch.ones(self.S, dtype=F64, device=dev))
        self.cnt, self.has_line, self.cnt_th = cnt[None, :, None], (cth > 0)[None, :, None], cth.clamp(min=1)[None, :, None]
        self.term_cnt = cnt
        act = torch.ones((Kp, L, 1), dtype=torch.bool, device=dev)
        for k, l in enumerate(net["outaged"], start=1):
            act[k, int(l)] = False
        self.act = act
        # parameters reach the kernels as FP32 values
        p = params or {}
        q = lambda a: f(np.asarray(a, np.float32))
        self.b = q(net["line_b"])[None, :, None]
        self.u_lim = p.get("line_u", q(net["line_u"]))
        self.load_p = p.get("load_p", q(net["load_p"]))
        self.pmax = p.get("gen_pmax", q(net["gen_pmax"]))
        self.pmin, self.a, self.gb = q(net["gen_pmin"]), q(net["gen_a"])[:, None], q(net["gen_b"])[:, None]
        self.voll = q(net["load_voll"])[:, None]
        self.hvdc_u = q(net["hvdc_u"])[:, None]
        ramp = np.asarray(net["gen_ramp"])
        self.ri = i(np.nonzero((ramp >= 0) & (T > 1))[0])
        if len(self.ri):
            self.rA = _ramp_rows(T).to(dev)
            R = q(ramp)[self.ri][:, None].expand(-1, 2 * (T - 1))
            self.rh = torch.cat([self.pmax[self.ri], -self.pmin[self.ri], R], 1)
            self.r_lam = torch.zeros((len(self.ri), len(self.rA)), dtype=F64, device=dev)
            self.r_bet = self.r_lam.clone()
        if self.B:
            eff, P = np.asarray(net["stor_eff"], np.float32), q(net["stor_P"])[:, None]
            if len(set(eff.tolist())) != 1:
                raise ValueError("one efficiency for every battery")
            A, eq = _battery_rows(T, float(eff[0]))
            self.sA, self.s_eq = A.to(dev), eq.to(dev)
            one, zero = torch.ones((self.B, T), dtype=F64, device=dev), torch.zeros((self.B, T), dtype=F64, device=dev)
            E = q(net["stor_dur"])[:, None] * P
            z1 = torch.zeros((self.B, T + 1), dtype=F64, device=dev)
            self.sh = torch.cat([zero, zero, zero[:, :1], zero[:, :1], P * one, zero, P * one, zero, E + z1, z1], 1)
            self.scost = q(net["stor_cost"])[:, None]
            self.sq = torch.zeros((self.B, 4 * T + 1), dtype=F64, device=dev)
            self.sq[:, 2 * T:3 * T] = self.scost
            self.s_lam = torch.zeros((self.B, 8 * T + 4), dtype=F64, device=dev)
            self.s_bet = self.s_lam.clone()
            self.s_z = self.sq.new_zeros(self.sq.shape)
        self._rho = None
        zl = torch.zeros((Kp, 2 * L, T), dtype=F64, device=dev)
        self.p, self.th, self.v, self.z, self.xi = zl, zl, zl, zl, zl
        self.pd = torch.zeros((self.S, T), dtype=F64, device=dev)
        self.zd = torch.zeros((Kp, self.S, T), dtype=F64, device=dev)
        self.u = torch.zeros((Kp, N, T), dtype=F64, device=dev)

    def _mean(self, line, dev=None):
        s = torch.zeros((self.Kp, self.N, self.T), dtype=F64, device=self.dev).index_add(1, self.line_node, line)
        if dev is None:
            return torch.where(self.has_line, s / self.cnt_th, torch.zeros_like(s))
        return s.index_add(1, self.dev_node, dev) / self.cnt

    def load_state(self, st):
        f = lambda k: st[k].to(self.dev, F64)
        p = f("p_line")
        half = torch.where(self.act, p / (2 * self.b), 0.5 * (f("th1") - f("th2")))
        mid = 0.5 * (f("th1") + f("th2"))
        self.p = torch.cat([-p, p], 1)
        self.th = torch.cat([mid + half, mid - half], 1)
        v = torch.cat([f("v1"), f("v2")], 1)
        self.v = v - self._mean(v)[:, self.line_node]
        self.pd, self.u = f("p_dev"), f("u")
        pbar = self._mean(self.p, self.pd[None].expand(self.Kp, -1, -1))
        self.z, self.zd = self.p - pbar[:, self.line_node], self.pd[None] - pbar[:, self.dev_node]
        self.xi = self._mean(self.th)[:, self.line_node]
        inner, T = f("inner"), self.T
        n = len(self.ri) * 2 * (4 * T - 2)
        if len(self.ri):
            r = inner[:n].reshape(len(self.ri), 2, -1)
            self.r_lam, self.r_bet = r[:, 0].clone(), r[:, 1].clone()
        if self.B:
            s = inner[n:].reshape(self.B, 2, -1)
            self.s_lam, self.s_bet = s[:, 0].clone(), s[:, 1].clone()

    def state(self):
        L = self.L
        inner = [torch.zeros(0, dtype=F64, device=self.dev)]
        if len(self.ri):
            inner.append(torch.stack([self.r_lam, self.r_bet], 1).reshape(-1))
        if self.B:
            inner.append(torch.stack([self.s_lam, self.s_bet], 1).reshape(-1))
        return dict(p_line=self.p[:, L:], th1=self.th[:, :L], th2=self.th[:, L:], v1=self.v[:, :L], v2=self.v[:, L:],
                    p_dev=self.pd, u=self.u, inner=torch.cat(inner))

    def _inner(self, x, A, h, eq, q, rho, minv, bet, lam):
        n = x.shape[1]
        for _ in range(10):
            rhs = rho * ((h + bet - lam) @ A) - q
            rhs = torch.cat([rhs[:, :n] + rho * x, rhs[:, n:]], 1)
            z = rhs @ minv if minv.dim() == 2 else torch.einsum("dij,dj->di", minv, rhs)
            al = z @ A.T - h
            nb = torch.clamp(al + lam, max=0.0)
            bet = nb if eq is None else torch.where(eq, torch.zeros_like(nb), nb)
            lam = lam + al - bet
        return z, bet, lam

    def _devices(self, X):
        G, D, B, T, rho = self.G, self.D, self.B, self.T, self.Kp * self.rho_p
        if self._rho != rho:
            self._rho = rho
            if len(self.ri):
                M = rho * (self.rA.T @ self.rA) + rho * torch.eye(T, dtype=F64, device=self.dev)
                self.r_inv = torch.linalg.inv(M[None] + 2 * self.a[self.ri][:, :, None] *
                                              torch.eye(T, dtype=F64, device=self.dev)[None])
            if B:
                M = rho * (self.sA.T @ self.sA)
                M[:T, :T] += rho * torch.eye(T, dtype=F64, device=self.dev)
                self.s_inv = torch.linalg.inv(M)
        parts = []
        pg = torch.clamp((rho * X[:G] - self.gb) / (2 * self.a + rho), min=self.pmin, max=self.pmax)
        if len(self.ri):
            z, self.r_bet, self.r_lam = self._inner(X[self.ri], self.rA, self.rh, None, self.gb[self.ri], rho,
                                                    self.r_inv, self.r_bet, self.r_lam)
            pg = pg.index_put((self.ri,), z)
        parts.append(pg)
        pl = torch.clamp((rho * X[G:G + D] - self.voll) / rho, min=-self.load_p, max=torch.zeros_like(self.load_p))
        parts.append(torch.where(self.voll < 0, -self.load_p, pl))
        if B:
            z, self.s_bet, self.s_lam = self._inner(X[G + D:G + D + B], self.sA, self.sh, self.s_eq, self.sq, rho,
                                                    self.s_inv, self.s_bet, self.s_lam)
            self.s_z = z
            parts.append(z[:, :T])
        if self.H:
            xh = X[G + D + B:].reshape(self.H, 2, T)
            p2 = torch.clamp((xh[:, 1] - xh[:, 0]) / 2, min=-self.hvdc_u, max=self.hvdc_u)
            parts.append(torch.stack([-p2, p2], 1).reshape(2 * self.H, T))
        return torch.cat(parts)

    def step(self, residuals=True):
        L, al, rp, rt, ln, dn = self.L, self.alpha, self.rho_p, self.rho_th, self.line_node, self.dev_node
        z, zd, xi, v, u, act, b = self.z, self.zd, self.xi, self.v, self.u, self.act, self.b
        x, y = z - u[:, ln], xi - v
        x1, x2, y1, y2 = x[:, :L], x[:, L:], y[:, :L], y[:, L:]
        ul = self.u_lim[None, :, None]
        p2 = torch.clamp((rp * (x2 - x1) + rt * (y1 - y2) / (2 * b)) / (2 * rp + rt / (2 * b * b)), min=-ul, max=ul)
        mid = 0.5 * (y1 + y2)
        th = torch.cat([torch.where(act, mid + p2 / (2 * b), y1), torch.where(act, mid - p2 / (2 * b), y2)], 1)
        p2 = torch.where(act, p2, torch.zeros_like(p2))
        p = torch.cat([-p2, p2], 1)
        pd = self._devices((zd - u[:, dn]).mean(0))
        ph, pdh, thh = al * p + (1 - al) * z, al * pd[None] + (1 - al) * zd, al * th + (1 - al) * xi
        wl, wd = ph + u[:, ln], pdh + u[:, dn]
        un = self._mean(wl, wd)
        zn, zdn = wl - un[:, ln], wd - un[:, dn]
        xin = self._mean(thh + v)[:, ln]
        vn = v + thh - xin
        self.it += 1
        if residuals and self.adapt_every and self.it % self.adapt_every == 0:
            sq = lambda *a: math.sqrt(sum(float((t * t).sum()) for t in a))
            r_pp, r_pt = sq(p - zn, pd[None] - zdn), sq(th - xin)
            r_dp, r_dt = rp * sq(zn - z, zdn - zd), rt * sq(xin - xi)
            for name, pr, du in (("rho_p", r_pp, r_dp), ("rho_th", r_pt, r_dt)):
                old = getattr(self, name)
                new = old * 1.1 if pr > 2 * du else old / 1.1 if du > 2 * pr else old
                if new == old:
                    continue
                setattr(self, name, new)
                if name == "rho_th":
                    vn = vn * (old / new)
                    continue
                un = un * (old / new)
                if len(self.ri):
                    self.r_lam = self.r_lam * (old / new)
                if self.B:
                    self.s_lam = self.s_lam * (old / new)
        self.p, self.th, self.pd, self.z, self.zd, self.xi, self.u, self.v = p, th, pd, zn, zdn, xin, un, vn

    def theta_node(self):
        """Node means of the line angles."""
        return self._mean(self.th)

    def objective(self):
        G, D, T = self.G, self.D, self.T
        pg, pl = self.pd[:G], self.pd[G:G + D]
        f = (self.a * pg * pg + self.gb * pg).sum()
        f = f + torch.where(self.voll < 0, torch.zeros_like(pl), self.voll * (pl + self.load_p)).sum()
        if self.B:
            f = f + (self.scost * self.s_z[:, 2 * T:3 * T]).sum()
        return f


def _solution(r):
    return dict(p_dev=r.pd, p_line=r.p[:, r.L:], theta_node=r.theta_node(), price=-r.rho_p * r.u.sum(0))


def _exact_net(case, seed):
    net, X, Y, flat = _net_inputs(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    N, T, F = net["n_nodes"], net["T"], case["F"]
    shapes = [(F, 64), (64,)] + [(64, 64), (64, 64), (64,)] * 3 + [(64, 2), (2,)]
    w, o = [], 0
    for shp in shapes:
        n = int(np.prod(shp))
        t = torch.from_numpy(flat[o:o + n].reshape(shp).copy())
        # matrices are used rounded to bfloat16
        w.append((t.to(torch.bfloat16) if len(shp) == 2 else t).to(dev, F64).requires_grad_(True))
        o += n
    lf, lt = (torch.as_tensor(net[k], dtype=torch.long, device=dev) for k in ("line_from", "line_to"))
    b = torch.as_tensor(net["line_b"], dtype=F64, device=dev)
    bs = torch.zeros(N, dtype=F64, device=dev).index_add(0, lf, b).index_add(0, lt, b)
    wf, wt = (b / bs[lf]).float().to(F64)[None, :, None], (b / bs[lt]).float().to(F64)[None, :, None]

    def average(H):
        H = H.reshape(T, N, 64)
        s = torch.zeros_like(H).index_add(1, lf, wf * H[:, lt]).index_add(1, lt, wt * H[:, lf])
        return s.reshape(T * N, 64)

    x, yt = (torch.from_numpy(a).to(dev, F64) for a in (X, Y))
    h = torch.relu(x @ w[0] + w[1])
    for l in range(3):
        h = torch.relu(h @ w[2 + 3 * l] + average(h) @ w[3 + 3 * l] + w[4 + 3 * l])
    y = h @ w[-2] + w[-1]
    loss = (torch.tensor(NET_SCALE, dtype=F64, device=dev) * (y - yt) ** 2).sum() / (N * T)
    g = torch.autograd.grad(loss, w)
    return dict(loss=float(loss), grad=torch.cat([t.reshape(-1) for t in g]).cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "net":
        return _exact_net(case, seed)
    if kind == "grad":
        net = _instance(case, seed)
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        prm = {k: torch.as_tensor(np.asarray(net[k], np.float32), device=dev).to(F64).requires_grad_(True)
               for k in ("load_p", "gen_pmax", "line_u")}
        r = _Iteration(net, params=prm, adapt_every=0)
        for _ in range(case["iters"]):
            r.step()
        f = r.objective()
        g = torch.autograd.grad(f, list(prm.values()), allow_unused=True)
        return dict({k: torch.zeros_like(prm[k]) if t is None else t for k, t in zip(prm, g)}, cost=float(f.detach()))
    with torch.no_grad():
        if kind == "batch":
            outs = []
            for net in _batch_instances(case, seed):
                r = _Iteration(net)
                for _ in range(case["iters"]):
                    r.step()
                outs.append(_solution(r))
            return outs
        if kind == "resolve":
            st, rho_p, rho_th = _previous(case["config"], case["n_nodes"], case["T"], case["K"])
            r = _Iteration(_instance(case, seed), rho_p=rho_p, rho_th=rho_th)
            r.load_state(st)
            for _ in range(case["iters"]):
                r.step()
            return r.state()
        r = _Iteration(_instance(case, seed), alpha=case["alpha"])
        for _ in range(case["iters"]):
            r.step()
        return dict(_solution(r), objective=float(r.objective()))
