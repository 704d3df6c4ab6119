"""The work a user of this solver has it do, as cases that can be timed and compared.

A case is one call of the public interface (``paper_2512_06715_gb300.pdhg``) on a seeded unit-commitment
relaxation: a capped solve of one LP, a batch of branch-and-bound node LPs, the rescaled products K v and K^T v
on their own, or the gradient of the optimal cost.  Sizes are the networks and horizons of ``instances.WORKLOADS``
(the 24-bus parity case up to the 6717-bus bench workload); ``draw`` spreads over the same range with odd sizes.

Two step rules are used, both plain solver options, because a long adaptive solve amplifies the rounding of its
own step-size sums until two correct runs no longer agree:
* "settled":  the adaptive rule, restarts, primal weight and refinement folds, with the growth of the step switched
  to the value it has late in a long solve (next to none);
* "constant": the textbook iteration with constant steps.
Solves are capped at a number of attempts, as the bench caps them; a mixed-precision point is handed on in FP32,
the precision of its iterates.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_06715_gb300 import pdhg
from paper_2512_06715_gb300.instances import VAR_SHED, build_instance, node_fixings

TOL = 1e-12          # never reached here: every solve runs to its cap of attempts
SETTLED = dict(step_growth_exp=8.0)  # (k+1)^-8: the step no longer grows after the first attempts
CONSTANT_STEP = 0.9  # the rescaled matrix has 2-norm <= 1, so constant steps below 1 are stable


def _net(buses, lines, gens, periods, slack=False):
    return dict(buses=buses, lines=lines, gens=gens, periods=periods, slack=slack)


def listed():
    return [
        # the smallest day: a teaching-size network re-solved often, where latency and launches count
        dict(name="day24_fp64", kind="solve", **_net(24, 38, 33, 24), precision="fp64", steps="constant", attempts=512),
        dict(name="day24_mixed", kind="solve", **_net(24, 38, 33, 24), precision="mixed", steps="settled",
             attempts=1024),
        # a day in 18 steps on the 4224-bus network, in full FP64 (bounds that are quoted)
        dict(name="day4224_T18_fp64", kind="solve", **_net(4224, 5900, 600, 18), precision="fp64", steps="settled",
             attempts=512),
        # the 4224-bus day in half hours: the ordinary mixed-precision relaxation
        dict(name="day4224_T48_mixed", kind="solve", **_net(4224, 5900, 600, 48), precision="mixed", steps="settled",
             attempts=512),
        # the 6049-bus network in 42 steps (no multiple of a warp), constant steps
        dict(name="day6049_T42_mixed", kind="solve", **_net(6049, 8470, 850, 42), precision="mixed",
             steps="constant", attempts=512),
        # the largest: the 6717-bus day in quarter hours, in both precisions (the bench workload)
        dict(name="day6717_T96_mixed", kind="solve", **_net(6717, 9200, 1000, 96), precision="mixed",
             steps="settled", attempts=512),
        dict(name="day6717_T96_fp64", kind="solve", **_net(6717, 9200, 1000, 96), precision="fp64", steps="settled",
             attempts=512),
        # node LPs of a branch and bound: a few open nodes of a small tree, a full batch on a 200-bus network, a
        # full batch on the 6049-bus network
        dict(name="nodes24_x9", kind="nodes", **_net(24, 38, 33, 24, True), nodes=9, attempts=512),
        dict(name="nodes200_x64", kind="nodes", **_net(200, 300, 60, 24, True), nodes=64, attempts=512),
        dict(name="nodes6049_x64", kind="nodes", **_net(6049, 8470, 850, 48, True), nodes=64, attempts=64),
        # the rescaled matrix applied to a vector, both ways, FP64 and FP32 (warm starts, residuals of other points)
        dict(name="products4224_T48", kind="products", **_net(4224, 5900, 600, 48)),
        # backward: the gradient of the optimal cost with respect to loads and costs (nodal prices) after a solve
        dict(name="prices4224_T18", kind="prices", **_net(4224, 5900, 600, 18)),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _drawn_net(rng, most_buses, most_periods, slack):
    buses = _log_uniform(rng, 24, most_buses)
    lines = int(buses * rng.uniform(1.36, 1.58))
    gens = max(5, int(buses * rng.uniform(0.12, 0.22)))
    return _net(buses, lines, gens, _log_uniform(rng, 12, most_periods), slack)


def draw(rng):
    most = max(work(c)["bytes"] for c in listed())
    while True:
        kind = rng.choice(("solve", "solve", "solve", "solve", "nodes", "nodes", "products", "prices"))
        if kind == "solve":
            case = dict(kind=kind, **_drawn_net(rng, 6717, 96, rng.random() < 0.25),
                        precision=rng.choice(("fp64", "mixed")), steps=rng.choice(("settled", "settled", "constant")),
                        attempts=64 * _log_uniform(rng, 2, 8))
        elif kind == "nodes":
            case = dict(kind=kind, **_drawn_net(rng, 3000, 48, True), nodes=_log_uniform(rng, 2, 64),
                        attempts=64 * _log_uniform(rng, 1, 4))
        else:
            case = dict(kind=kind, **_drawn_net(rng, 6717, 96, rng.random() < 0.25))
        if work(case)["bytes"] <= most:
            return case


def _instance(case, seed):
    """The relaxation of one day on the case's network: the network is the same every day, the loads and the offers
    (costs) are the seed's."""
    inst = build_instance(case["buses"], case["lines"], case["gens"], case["periods"], with_slack=case["slack"])
    rng = np.random.default_rng(seed)
    level = rng.uniform(0.85, 1.0, (inst.n_periods, 1)) * rng.uniform(0.97, 1.03, inst.load.shape)
    inst.load = inst.load * level
    inst.q[inst.row_balance] = inst.load
    inst.c *= rng.uniform(0.9, 1.1, inst.n)
    if case["slack"]:  # no more can be shed than is asked for
        inst.u[inst.var_kind == VAR_SHED] = inst.load.reshape(-1)
    return inst


def prepare(case, seed):
    """A workspace that has solved once, as a program that solves day after day keeps it: device copy of the LP,
    layout, launch shapes, graph.  Solves start cold every time."""
    inst = _instance(case, seed)
    kind = case["kind"]
    state = dict(kind=kind)
    if kind in ("solve", "prices"):
        precision = case.get("precision", "fp64")
        opts = dict(precision=precision, tol=TOL, max_iters=case.get("attempts", 256))
        if case.get("steps") != "constant":
            opts.update(SETTLED)
        ws = pdhg.Workspace.from_instance(inst, pdhg.default_opts(**opts))
        if case.get("steps") == "constant":
            ws.prepare()
            dr, dc = ws.scaling()
            ws.set_opts(fixed_eta=CONSTANT_STEP, fixed_omega=float((dc * ws.t["c"]).norm() / (dr * ws.t["q"]).norm()))
        ws.solve()
        state.update(ws=ws, precision=precision)
    elif kind == "nodes":
        l_b, u_b = node_fixings(inst, case["nodes"], seed0=1000 + seed % 100000)
        ws = pdhg.Workspace.from_instance(inst, pdhg.default_opts(precision="mixed", tol=TOL,
                                                                  max_iters=case["attempts"], **SETTLED))
        l_b, u_b = (torch.as_tensor(b, device=ws.device) for b in (l_b, u_b))
        ws.solve_batched(l_b, u_b)
        state.update(ws=ws, l=l_b, u=u_b)
    else:
        ws = pdhg.Workspace.from_instance(inst)
        ws.prepare()
        state["ws"] = ws
        state["x"], state["y"] = (v.to(ws.device) for v in _product_inputs(inst, seed))
    return state


def _product_inputs(inst, seed):
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(inst.n, generator=g, dtype=torch.float64),
            torch.randn(inst.m, generator=g, dtype=torch.float64))


def run(state):
    ws, kind = state["ws"], state["kind"]
    if kind == "solve":
        x, y, r = ws.solve()
        if state["precision"] == "mixed":
            x, y = x.float(), y.float()
        return dict(x=x, y=y, rel_kkt=r["rel_kkt"], attempts=r["iterations"])
    if kind == "nodes":
        x, y, r = ws.solve_batched(state["l"], state["u"])
        return dict(x=x.float(), y=y.float(), rel_kkt=np.array([k["rel_kkt"] for k in r], np.float32),
                    attempts=np.array([k["iterations"] for k in r]))
    if kind == "products":
        kx = ws.apply_K(state["x"])
        kty = ws.apply_K(state["y"], transpose=True)
        kx32 = ws.apply_K(state["x"], precision=pdhg.PREC_MIXED)
        kty32 = ws.apply_K(state["y"], transpose=True, precision=pdhg.PREC_MIXED)
        return dict(kx=kx, kty=kty, kx32=kx32.float(), kty32=kty32.float())
    # the C entry point that UCRelax's backward calls, with the cotangent of the cost alone
    grad_q = torch.empty(ws.m, dtype=torch.float64, device=ws.device)
    grad_c = torch.empty(ws.n, dtype=torch.float64, device=ws.device)
    pdhg._check(pdhg.lib().pdhg_backward(ws.ws, 1.0, None, grad_q.data_ptr(), grad_c.data_ptr(),
                                         torch.cuda.current_stream(ws.device).cuda_stream), "pdhg_backward")
    return dict(grad_q=grad_q, grad_c=grad_c)


def _sizes(case):
    """Columns, rows and nonzeros of the relaxation, estimated from the network (exact but for the nonzeros of the
    balance rows and of the minimum up/down rows)."""
    N, L, G, T = case["buses"], case["lines"], case["gens"], case["periods"]
    n = T * (4 * G + N) + (T * (N + min(N, G)) if case["slack"] else 0)
    m = T * N + 2 * T * L + 2 * T * G + 5 * (T - 1) * G
    window = min(T, max(1.0, 4.0 * T / 24.0))  # minimum up/down times of 2 to 6 hours
    nnz = T * (N + 2 * L + G) + 4 * T * L + 4 * T * G + 12 * (T - 1) * G + 2 * (T - 1) * G * (1 + window)
    return n, m, nnz + (2 * T * N if case["slack"] else 0)


def work(case):
    """Bytes and operations one pass cannot do without.  Per attempt: the matrix values once per product, the row
    vectors y, q, y_lo, y-average read and y', y-average written, the column vectors x, c, l, u, x-average read and
    x', x-average, K^T y written; the positions of the entries are structure and not counted."""
    n, m, nnz = _sizes(case)
    kind = case["kind"]
    if kind in ("products", "prices"):
        # products: values, input and output of four products; prices: solution and scaling in, gradients out
        b = (2 * nnz * 8 + 2 * nnz * 4 + 4 * 8 * (n + m)) if kind == "products" else 3 * 8 * (n + m)
        return dict(bytes=float(b), flops=float(8 * nnz if kind == "products" else 2 * (n + m)))
    per_vector, per_value, width = (4, 4, case["nodes"]) if kind == "nodes" else \
        ((8, 8, 1) if case["precision"] == "fp64" else (4, 4, 1))
    k = case["attempts"]
    attempt = 2 * nnz * per_value + width * per_vector * (6 * m + 8 * n)
    check = 2 * nnz * 8 + width * 8 * (4 * m + 6 * n)
    flops = width * (k * (4 * nnz + 10 * m + 8 * n) + (k // 64) * (8 * nnz + 40 * m + 50 * n))
    return dict(bytes=float(k * attempt + (k // 64) * check + width * 16 * (n + m)), flops=float(flops))


# ---- 64-bit values ------------------------------------------------------------------------------------------------

class _Scaled:
    """The LP of an instance on the GPU in 64 bits with its Ruiz (10 passes) and Pock-Chambolle factors."""

    def __init__(self, inst):
        t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
        self.n, self.m, self.m_eq = inst.n, inst.m, inst.m_eq
        rp = t(inst.row_ptr)
        self.row = torch.repeat_interleave(torch.arange(inst.m, device="cuda"), rp[1:] - rp[:-1])
        self.col = t(inst.col).long()
        val = t(inst.val)
        self.dr = torch.ones(inst.m, dtype=torch.float64, device="cuda")
        self.dc = torch.ones(inst.n, dtype=torch.float64, device="cuda")
        for p in range(11):
            a = (val * self.dr[self.row] * self.dc[self.col]).abs()
            how = "amax" if p < 10 else "sum"
            r = torch.zeros_like(self.dr).scatter_reduce_(0, self.row, a, how)
            c = torch.zeros_like(self.dc).scatter_reduce_(0, self.col, a, how)
            self.dr = self.dr * torch.where(r > 0, r.rsqrt(), torch.ones_like(r))
            self.dc = self.dc * torch.where(c > 0, c.rsqrt(), torch.ones_like(c))
        val = val * self.dr[self.row] * self.dc[self.col]
        self.k = torch.sparse_csr_tensor(rp, self.col, val, size=(inst.m, inst.n))
        order = torch.argsort(self.col, stable=True)
        cp = torch.zeros(inst.n + 1, dtype=torch.int64, device="cuda")
        cp[1:] = torch.cumsum(torch.bincount(self.col, minlength=inst.n), 0)
        self.kt = torch.sparse_csr_tensor(cp, self.row[order], val[order], size=(inst.n, inst.m))
        self.c0, self.q0 = t(inst.c), t(inst.q)
        self.c, self.q = self.c0 * self.dc, self.q0 * self.dr
        self.l, self.u = t(inst.l) / self.dc, t(inst.u) / self.dc
        self.ineq = torch.arange(inst.m, device="cuda") >= inst.m_eq

    def rel_kkt(self, x, y):
        """Relative optimality error of a point, on the unscaled LP."""
        rp = self.q - self.k @ x
        rp = torch.where(self.ineq, rp.clamp(min=0), rp) / self.dr
        lam = self.c - self.kt @ y
        zero = torch.zeros_like(lam)
        lf, uf = torch.isfinite(self.l), torch.isfinite(self.u)
        pos, neg = torch.where(lf, lam.clamp(min=0), zero), torch.where(uf, lam.clamp(max=0), zero)
        rd = (lam - pos - neg) / self.dc
        primal = float(self.c @ x)
        dual = float(self.q @ y + (torch.where(lf, self.l, zero) * pos).sum() + (torch.where(uf, self.u, zero) * neg).sum())
        gap = abs(primal - dual) / (1 + abs(primal) + abs(dual))
        return max(float(rp.norm() / (1 + self.q0.norm())), float(rd.norm() / (1 + self.c0.norm())), gap)


def exact(case, seed):
    """64-bit values of the products and of the constant-step solves.  The other solves have none of their own: their
    accept, restart and fold decisions are part of the result."""
    kind = case["kind"]
    if kind == "products":
        inst = _instance(case, seed)
        lp = _Scaled(inst)
        x, y = (v.cuda() for v in _product_inputs(inst, seed))
        kx, kty = lp.k @ x, lp.kt @ y
        return dict(kx=kx, kty=kty, kx32=kx, kty32=kty)
    if kind != "solve" or case["steps"] != "constant":
        return None
    lp = _Scaled(_instance(case, seed))
    omega = float(lp.c.norm() / lp.q.norm())
    tau, sigma = CONSTANT_STEP / omega, CONSTANT_STEP * omega
    x = torch.zeros(lp.n, dtype=torch.float64, device="cuda").clamp(lp.l, lp.u)
    y = torch.zeros(lp.m, dtype=torch.float64, device="cuda")
    xs, ys, kx = torch.zeros_like(x), torch.zeros_like(y), lp.k @ x
    for _ in range(case["attempts"]):
        x = (x - tau * (lp.c - lp.kt @ y)).clamp(lp.l, lp.u)
        kn = lp.k @ x
        y = y + sigma * (lp.q - 2 * kn + kx)
        y = torch.where(lp.ineq, y.clamp(min=0), y)
        kx, xs, ys = kn, xs + x, ys + y
    xs, ys = xs / case["attempts"], ys / case["attempts"]
    if lp.rel_kkt(xs, ys) < lp.rel_kkt(x, y):  # the better of the last iterate and the average is returned
        x, y = xs, ys
    return dict(x=lp.dc * x, y=lp.dr * y, rel_kkt=None, attempts=None)
