"""What this framework is timed on: its evaluations, adjoint products and linear solves, as a
solver or a study calls them, through the public binding (paper_2203_10587_gb300.exago).

A case is a dict of plain values.  Common keys: "kind" (which call), "grid" (seed of the synthetic
grid), "nb" / "nl" / "ng" (its buses, branches, generators), "deg" (largest bus degree), "shift"
(share of phase-shifting transformers), "B" (states of the batch).  Kinds:

  polar / cart   the evaluation in polar or rectangular voltages; "states" says how the batch
                 comes about (one, n1, load, gen), "want" which outputs (all: an interior-point
                 iteration; trial: f and g | h alone, a line-search point)
  adjoint        J u, J'v and (hess L) u of the polar model, without forming J or H
  kkt            the interior-point KKT step of every state
  pflow          one power-flow Newton step of every state
  rows           what a security-constrained study adds to an evaluation: feasibility slacks, and
                 the ramp rows that couple the states, with their transpose products

Grids and batches come from the package's own seeded generator (synth); `exact` evaluates the
model a second time in plain torch, in 64 bits, from the textbook formulas.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2203_10587_gb300 import exago, synth

F64 = torch.float64


def listed():
    n2000 = {"grid": 3, "nb": 2000, "nl": 2700, "ng": 500, "deg": 8, "shift": 0.0}
    n10k = {"grid": 2, "nb": 10000, "nl": 13000, "ng": 2500, "deg": 8, "shift": 0.0}
    n200 = {"grid": 19, "nb": 200, "nl": 260, "ng": 50, "deg": 8, "shift": 0.0}
    return [
        # the smallest call: one interior-point iteration's evaluation of one small grid
        {"name": "polar_30_x1", "kind": "polar", "states": "one", "want": "all", "grid": 1,
         "nb": 30, "nl": 41, "ng": 6, "deg": 8, "shift": 0.0, "B": 1},
        # one large grid, one state: a single AC-OPF solved by itself
        {"name": "polar_10k_x1", "kind": "polar", "states": "one", "want": "all", **n10k, "B": 1},
        # the N-1 security study, every contingency's model in one call: the benchmark's workload
        {"name": "polar_2000_x512_n1", "kind": "polar", "states": "n1", "want": "all", **n2000,
         "B": 512},
        # a stochastic study: load scenarios of a large grid
        {"name": "polar_10k_x64_load", "kind": "polar", "states": "load", "want": "all", **n10k,
         "B": 64},
        # a meshed grid (six branches a bus) with phase shifters, under generator and branch outages
        {"name": "polar_meshed_x301_gen", "kind": "polar", "states": "gen", "want": "all",
         "grid": 7, "nb": 2000, "nl": 6000, "ng": 500, "deg": 16, "shift": 0.1, "B": 301},
        # line-search points of the paper's 200-bus study with 100 contingencies: values only
        {"name": "trial_200_x100_n1", "kind": "polar", "states": "n1", "want": "trial", **n200,
         "B": 100},
        # the N-1 study in rectangular voltages
        {"name": "cart_2000_x512_n1", "kind": "cart", "states": "n1", "want": "all", **n2000,
         "B": 512},
        # matrix-free iterations and automatic differentiation over load scenarios
        {"name": "adjoint_10k_x64", "kind": "adjoint", "states": "load", **n10k, "B": 64},
        # the linear solve of an interior-point iteration: the N-1 study, and a small one
        {"name": "kkt_2000_x512", "kind": "kkt", "states": "n1", **n2000, "B": 512},
        {"name": "kkt_200_x37", "kind": "kkt", "states": "n1", **n200, "B": 37},
        # a power-flow iteration of many dispatches
        {"name": "pflow_2000_x512", "kind": "pflow", "grid": 33, "nb": 2000, "nl": 2700,
         "ng": 500, "deg": 8, "shift": 0.0, "B": 512},
        # slacks and ramp rows of the N-1 study (contingencies tied to the base case)
        {"name": "rows_2000_x512_star", "kind": "rows", "tie": "star", **n2000, "B": 512},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["polar", "polar", "polar", "cart", "adjoint", "kkt", "pflow", "rows"])
    solve = kind in ("kkt", "pflow")
    nb = log_int(30, 2000 if solve else 10000)
    mesh = 1.35 if solve or nb > 2000 else rng.choice([1.35, 1.35, 3.0])
    nl = int(nb * rng.uniform(1.2, mesh))
    c = {"kind": kind, "grid": rng.randrange(1, 10000), "nb": nb, "nl": nl,
         "ng": max(2, int(nb * rng.uniform(0.1, 0.3))), "deg": 8 if mesh < 2 else 16,
         "shift": rng.choice([0.0, 0.0, 0.1]),
         "B": log_int(1, max(1, min(512, 2700 * 512 // max(nl, 2700), 1350000 // nl)))}
    if kind in ("polar", "cart"):
        c["states"] = rng.choice(["one", "n1", "load", "gen"])
        c["want"] = rng.choice(["all", "all", "trial"])
    elif kind in ("adjoint", "kkt"):
        c["states"] = rng.choice(["n1", "load"])
    elif kind == "rows":
        c["tie"] = rng.choice(["star", "chain"])
    return c


# ---- inputs -----------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _grid(seed, nb, nl, ng, deg, shift, light):
    g = synth.make_grid(seed, nb, nl, ng, max_degree=deg, shunts=not light and seed % 2 == 0,
                        transformer_frac=0.2 if light else 0.1, shifter_frac=shift)
    if light:   # loads at which a flat start converges
        g.Pd *= 0.3
        g.Qd *= 0.3
    return g


def grid_of(case):
    return _grid(case["grid"], case["nb"], case["nl"], case["ng"], case["deg"], case["shift"],
                 case["kind"] == "pflow")


@functools.lru_cache(maxsize=4)
def _outage_branches(seed, nb, nl, ng, deg, shift, light):
    g = _grid(seed, nb, nl, ng, deg, shift, light)
    return np.flatnonzero(~synth.bridges(g.nb, g.f, g.t))


def _batch(case, seed):
    """Host arrays of the batch: x, lambda (rectangular: with the voltage rows'), masks, scales."""
    g, B = grid_of(case), case["B"]
    rng = np.random.default_rng([seed, 17])
    x0, lam0 = synth.base_state(rng, g)
    b = {"mask": None, "gen_mask": None, "pd_scale": None, "weight": None}
    states = case["states"]
    x, lam = np.repeat(x0[None], B, 0), np.repeat(lam0[None], B, 0)
    if states != "load":
        x += rng.normal(0.0, 0.02, x.shape)
        lam += rng.normal(0.0, 0.02, lam.shape)
    if states == "load":
        b["pd_scale"] = np.exp(0.1 * rng.normal(size=(B, g.nb)))
        b["weight"] = np.full(B, 1.0 / B)
    if states in ("n1", "gen"):   # one branch that does not island a bus, and one generator
        cand = _outage_branches(case["grid"], case["nb"], case["nl"], case["ng"], case["deg"],
                                case["shift"], case["kind"] == "pflow")
        b["mask"] = np.ones((B, g.nl), np.uint8)
        if cand.size:
            b["mask"][np.arange(B), rng.choice(cand, size=B, replace=B > cand.size)] = 0
    if states == "gen":
        b["gen_mask"] = np.ones((B, g.ng), np.uint8)
        b["gen_mask"][np.arange(B), rng.integers(0, g.ng, B)] = 0
    if case["kind"] == "cart":
        va, vm = x[:, :g.nb].copy(), x[:, g.nb:2 * g.nb].copy()
        x[:, :g.nb], x[:, g.nb:2 * g.nb] = vm * np.cos(va), vm * np.sin(va)
        lam = np.concatenate([lam, rng.normal(size=(B, g.nb))], 1)
    b["x"], b["lam"] = x, lam
    return b


def _cuda(a):
    return None if a is None else torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _randn(seed, *shape):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(*shape, dtype=F64, device="cuda", generator=gen)


def _empty(*shape):
    return torch.empty(*shape, dtype=F64, device="cuda")


class _Owned:
    """A handle of the C interface that is given back with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def prepare(case, seed):
    g, kind, B = grid_of(case), case["kind"], case["B"]
    net = exago.Net(g)
    s = {"case": case, "net": net}
    if kind in ("polar", "cart", "adjoint"):
        b = _batch(case, seed)
        s["batch"] = exago.make_batch(_cuda(b["x"]), _cuda(b["lam"]), _cuda(b["mask"]),
                                      _cuda(b["pd_scale"]), _cuda(b["weight"]), 1.0,
                                      gen_mask=_cuda(b["gen_mask"]))
    if kind in ("polar", "cart"):
        full = case["want"] == "all"
        n, me, mi, nj, nh = (exago.exago_net_dims if kind == "polar"
                             else exago.exago_net_dims_cart)(net.h)
        s["out"] = {"f": _empty(B), "grad": _empty(B, n) if full else None,
                    "gh": _empty(B, me + mi), "jval": _empty(B, nj) if full else None,
                    "hval": _empty(B, nh) if full else None}
    elif kind == "adjoint":
        s["u"], s["v"] = _randn(seed, B, net.n), _randn(seed + 1, B, net.m)
        s["out"] = {"ju": _empty(B, net.m), "jtv": _empty(B, net.n), "hu": _empty(B, net.n)}
    elif kind == "kkt":
        s.update(_kkt_inputs(case, seed))
        s["kkt"] = _Owned(exago.exago_kkt_create(net.h), exago.exago_kkt_destroy)
        s["ws"] = torch.empty(exago.exago_kkt_workspace_size(s["kkt"].h, B), dtype=torch.uint8,
                              device="cuda")
        s["out"] = {"sol": torch.empty_like(s["rhs"]),
                    "inertia": torch.empty(B, 2, dtype=torch.int32, device="cuda")}
    elif kind == "pflow":
        x, types, scale = _pflow_inputs(case, seed)
        s["pf"] = _Owned(exago.exago_pf_create(net.h, types), exago.exago_pf_destroy)
        ws = torch.empty(exago.exago_pf_workspace_size(s["pf"].h, B), dtype=torch.uint8,
                         device="cuda")
        s["batch"] = exago.make_batch(_cuda(x), pd_scale=_cuda(scale), workspace=ws)
        s["out"] = {"x": _empty(B, net.n), "mismatch": _empty(B)}
    elif kind == "rows":
        r = _rows_inputs(case, seed)
        s.update({k: _cuda(r[k]) for k in ("x", "z", "gh", "v", "nu", "weight")})
        s["slack"] = exago.Slack(net, r["bus"], r["row"], r["sign"], r["cost"])
        s["tie"] = exago.Coupling(net, synth.coupling_parents(case["tie"], B))
        s["batch"] = exago.make_batch(s["x"], obj_weight=s["weight"])
        nz = s["slack"].nz
        # g | h and f arrive from the evaluation and the slacks are added in place: the call
        # here gets fresh copies of them each time, as an evaluation would have written them
        s["out"] = {"gh": torch.empty_like(s["gh"]), "f": _empty(B), "grad_z": _empty(B, nz),
                    "jtv_z": _empty(B, nz), "r": _empty(B, g.ng), "ct_nu": _empty(B, g.ng)}
    return s


def run(state):
    kind, net, out = state["case"]["kind"], state["net"], state["out"]
    if kind == "polar":
        exago.exago_eval_all(net.h, state["batch"], **out)
    elif kind == "cart":
        exago.exago_eval_cart(net.h, state["batch"], **out)
    elif kind == "adjoint":
        exago.exago_eval_jvp(net.h, state["batch"], state["u"], out["ju"])
        exago.exago_eval_jtv(net.h, state["batch"], state["v"], out["jtv"])
        exago.exago_eval_hvp(net.h, state["batch"], state["u"], out["hu"])
    elif kind == "kkt":
        exago.exago_kkt_solve(state["kkt"].h, state["jval"], state["hval"], state["dx"],
                              state["dc"], state["rhs"], out["sol"], out["inertia"], state["ws"])
    elif kind == "pflow":
        exago.exago_pf_step(state["pf"].h, state["batch"], out["x"], out["mismatch"])
    else:
        out["gh"].copy_(state["gh"])
        out["f"].zero_()
        exago.exago_eval_slack(state["slack"], state["batch"], state["z"], out["gh"], net.m,
                               out["f"], out["grad_z"])
        exago.exago_eval_slack_jtv(state["slack"], state["batch"], state["v"], net.m,
                                   out["jtv_z"])
        exago.exago_eval_coupling(state["tie"].h, state["x"], out["r"])
        exago.exago_eval_coupling_jtv(state["tie"].h, state["nu"], out["ct_nu"], net.ng)
    return {k: v for k, v in out.items() if v is not None}


def _kkt_inputs(case, seed):
    """J and the Lagrangian Hessian of the batch's states, the barrier's diagonals as an
    interior-point method regularises them (W + diag(dx) diagonally dominant), a right-hand side."""
    g, B = grid_of(case), case["B"]
    b = _batch(case, seed)
    M = Model(g, False)
    _, _, jval, hval = M.evaluate(_cuda(b["x"]), _cuda(b["lam"]), _cuda(b["mask"]),
                                  _cuda(b["gen_mask"]), _cuda(b["pd_scale"]),
                                  _cuda(b["weight"]), 1.0)[1:]
    rows, cols = M.h_row, M.h_col
    a = hval.abs()
    dx = torch.ones(B, g.n, dtype=F64, device="cuda")
    for i, keep in ((rows, torch.ones_like(rows, dtype=torch.bool)), (cols, rows != cols)):
        order = torch.argsort(i[keep], stable=True)
        at = torch.searchsorted(i[keep][order], torch.arange(g.n + 1, device="cuda"))
        c = torch.cat([torch.zeros(B, 1, dtype=F64, device="cuda"),
                       a[:, keep][:, order].cumsum(1)], 1)
        dx += c[:, at[1:]] - c[:, at[:-1]]
    rng = np.random.default_rng([seed, 23])
    return {"jval": jval, "hval": hval, "dx": dx, "dc": _cuda(rng.uniform(0.5, 2.0, (B, g.m))),
            "rhs": _cuda(rng.normal(size=(B, g.n + g.m)))}


def _pflow_inputs(case, seed):
    """Dispatches near a flat start: slack, PV and PQ buses, spread generation and load."""
    g, B = grid_of(case), case["B"]
    rng = np.random.default_rng([seed, 29])
    types = np.ones(g.nb, np.int32)
    types[g.gbus] = 2
    types[g.gbus[0]] = 3
    x = np.zeros((B, g.n))
    x[:, :g.nb] = rng.normal(0.0, 0.02, (B, g.nb)) * (types != 3)
    x[:, g.nb:2 * g.nb] = 1.0 + rng.normal(0.0, 0.01, (B, g.nb)) * (types == 1)
    x[:, 2 * g.nb:2 * g.nb + g.ng] = g.Pd.sum() / g.ng * rng.uniform(0.9, 1.1, (B, g.ng))
    return x, types, np.exp(0.1 * rng.normal(size=(B, g.nb)))


def _rows_inputs(case, seed):
    """An imbalance pair on every balance and load loss at the loaded buses."""
    g, B = grid_of(case), case["B"]
    rng = np.random.default_rng([seed, 31])
    every, load = np.arange(g.nb), np.flatnonzero(g.Pd > 0.3)
    bus = np.concatenate([np.tile(every, 4), load, load]).astype(np.int32)
    row = np.repeat([0, 0, 1, 1, 0, 1], [g.nb] * 4 + [load.size] * 2).astype(np.int32)
    sign = np.repeat([-1, 1, -1, 1, -1, -1], [g.nb] * 4 + [load.size] * 2).astype(np.int32)
    return {"bus": bus, "row": row, "sign": sign, "cost": np.full(bus.size, 500.0),
            "x": rng.normal(size=(B, g.n)), "z": 0.1 * rng.random((B, bus.size)),
            "gh": rng.normal(size=(B, g.m)), "v": rng.normal(size=(B, g.m)),
            "nu": rng.normal(size=(B, g.ng)), "weight": rng.uniform(0.1, 1.0, B)}


# ---- the work that a pass cannot do without -----------------------------------------------------

def work(case):
    nb, nl, ng, B, kind = case["nb"], case["nl"], case["ng"], case["B"], case["kind"]
    n, m = 2 * nb + 2 * ng, 2 * nb + 2 * nl
    nj, nh = 4 * nb + 16 * nl + 2 * ng, 3 * nb + 4 * nl + ng   # parallel branches merge: at most
    net = 8 * (11 * nl + 4 * nb + 4 * ng) + 4 * (2 * nl + ng)
    mask = (nl if case.get("states") in ("n1", "gen") else 0) + (
        ng if case.get("states") == "gen" else 0) + (
        8 * nb + 8 if case.get("states") == "load" else 0)
    if kind in ("polar", "cart"):
        mm, njj = (m, nj) if kind == "polar" else (m + nb, nj + 2 * nb)
        if case["want"] == "trial":
            return {"bytes": B * (8 * (n + 1 + mm) + mask) + net,
                    "flops": B * (46 * nl + 2 * nl + 8 * nb + 6 * ng)}
        per = 168 * nl + 7 * max(0, 2 * nl - nb) + 16 * nb + 12 * ng
        return {"bytes": B * (8 * (n + mm + 1 + n + mm + njj + nh) + mask) + net,
                "flops": B * per}
    if kind == "adjoint":   # three products, x read once, two directions
        return {"bytes": B * (8 * (n + m + n + m + m + n + n) + mask) + net,
                "flops": B * nl * (80 + 100 + 190)}
    if kind == "kkt":
        blocks, pairs = _symbolic(case)
        return {"bytes": B * 8 * (nj + nh + n + m + 2 * (n + m)),
                "flops": B * 2 * (64 * pairs + 80 * blocks)}
    if kind == "pflow":
        blocks, pairs = _symbolic(case)
        return {"bytes": B * 8 * (2 * n + nb + 1),
                "flops": B * (2 * (16 * pairs + 16 * blocks) + 100 * nl)}
    nz = 4 * nb + 2 * int((grid_of(case).Pd > 0.3).sum())
    return {"bytes": B * 8 * (nz * 3 + 2 * m + 2 * nb + 4 * ng + 2), "flops": B * 4 * nz}


def _symbolic(case):
    """Blocks of the factor and block products of a factorisation on a minimum-degree order."""
    _, nbrs = _min_degree(case)
    d = [len(x) for x in nbrs]
    return sum(d) + case["nb"], sum(k * (k + 1) // 2 for k in d)


def _min_degree(case):
    return _order(case["grid"], case["nb"], case["nl"], case["ng"], case["deg"], case["shift"],
                  case["kind"] == "pflow")


@functools.lru_cache(maxsize=4)
def _order(*key):
    g = _grid(*key)
    adj = [set() for _ in range(g.nb)]
    for a, c in zip(g.f.tolist(), g.t.tolist()):
        adj[a].add(c)
        adj[c].add(a)
    deg = np.array([len(a) for a in adj])
    order, nbrs = [], []
    for _ in range(g.nb):
        k = int(np.argmin(deg))
        ring = adj[k]
        for i in ring:
            adj[i] |= ring
            adj[i] -= {i, k}
            deg[i] = len(adj[i])
        deg[k] = g.nb + 1
        order.append(k)
        nbrs.append(sorted(ring))
    return order, nbrs


# ---- the same results in plain torch, in 64 bits ------------------------------------------------

class Model:
    """The AC-OPF model in polar or rectangular voltages, term by term: every branch end adds
    its injections, their derivatives and its part of the Lagrangian's second derivatives, and
    the terms of one row and column are summed.  Rows and columns in the exported order."""

    def __init__(self, g, cart):
        self.g, self.cart = g, cart
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
        ys = 1.0 / (g.r + 1j * g.x)
        tau = np.where(g.tap == 0, 1.0, g.tap)
        tr = tau * np.exp(1j * (g.shift if g.shift is not None else np.zeros(g.nl)))
        yff, ytt = (ys + 0.5j * g.b) / tau ** 2, ys + 0.5j * g.b
        yft, ytf = -ys / np.conj(tr), -ys / tr
        self.ends = [(t(g.f).long(), t(g.t).long(), t(yff.real), t(yff.imag), t(yft.real), t(yft.imag)),
                     (t(g.t).long(), t(g.f).long(), t(ytt.real), t(ytt.imag), t(ytf.real), t(ytf.imag))]
        nb, nl, ng, n = g.nb, g.nl, g.ng, g.n
        f, to, bus, gen = g.f.astype(np.int64), g.t.astype(np.int64), np.arange(nb), np.arange(ng)
        gb = g.gbus.astype(np.int64)
        # places of the J terms, in the order `evaluate` lists them
        rows, cols = [], []
        for u, v in ((f, to), (to, f)):
            for r0 in (0, nb):
                for c in (u, v, nb + u, nb + v):
                    rows.append(r0 + u), cols.append(c)
        for side in (0, 1):
            u, v = (f, to) if side == 0 else (to, f)
            for c in (u, v, nb + u, nb + v):
                rows.append(2 * nb + side * nl + np.arange(nl)), cols.append(c)
        for r0 in (0, nb):
            for c0 in (0, nb):
                rows.append(r0 + bus), cols.append(c0 + bus)
        rows += [gb, nb + gb]
        cols += [2 * nb + gen, 2 * nb + ng + gen]
        if cart:
            rows += [2 * nb + 2 * nl + bus] * 2
            cols += [bus, nb + bus]
        self.j_at, self.nj, self.j_row, self.j_col = self._places(rows, cols, n)
        # places of the Hessian terms: the lower triangle
        rows, cols = [], []
        for u, v in ((f, to), (to, f)):
            i = (u, v, nb + u, nb + v)
            for a in range(4):
                for b in range(a + 1):
                    rows.append(np.maximum(i[a], i[b])), cols.append(np.minimum(i[a], i[b]))
        rows += [bus, nb + bus, nb + bus, 2 * nb + gen]
        cols += [bus, bus, nb + bus, 2 * nb + gen]
        self.h_at, self.nh, self.h_row, self.h_col = self._places(rows, cols, n)

    @staticmethod
    def _places(rows, cols, n):
        key = np.concatenate(rows) * n + np.concatenate(cols)
        where, at = np.unique(key, return_inverse=True)
        order = np.argsort(at, kind="stable")   # terms of one place side by side, in term order
        start = np.searchsorted(at[order], np.arange(where.size))
        count = np.diff(np.append(start, at.size))
        t = lambda a: torch.as_tensor(a, device="cuda")
        return (t(order), t(start), t(count)), where.size, t(where // n), t(where % n)

    @staticmethod
    def _sum(terms, at):
        """Terms [B, k] summed by place, term after term (the same sums on every run)."""
        order, start, count = at
        v = torch.cat(terms, 1)
        out = v[:, order[start]].clone()
        for i in range(1, int(count.max())):
            more = torch.nonzero(count > i).reshape(-1)
            out[:, more] += v[:, order[start[more] + i]]
        return out

    def _at_bus(self, terms, bus):
        """Sums over the branch ends or generators at each bus: [B, k] -> [B, nb]."""
        key = np.concatenate([b.cpu().numpy() for b in bus] + [np.arange(self.g.nb)])
        _, at = np.unique(key, return_inverse=True)
        order = np.argsort(at, kind="stable")
        start = np.searchsorted(at[order], np.arange(self.g.nb))
        count = np.diff(np.append(start, at.size))
        t = lambda a: torch.as_tensor(a, device="cuda")
        zero = torch.zeros(terms[0].shape[0], self.g.nb, dtype=F64, device="cuda")
        return self._sum(terms + [zero], (t(order), t(start), t(count)))

    def _end(self, x, end):
        """P, Q of a branch end, their gradients in (u, v, nb + u, nb + v) and second derivatives
        as {(i, j): value}, i >= j."""
        u, v, gs, bs, gm, bm = end
        nb = self.g.nb
        if not self.cart:
            th, vu, vv = x[:, u] - x[:, v], x[:, nb + u], x[:, nb + v]
            c, s = torch.cos(th), torch.sin(th)
            A, C = gm * c + bm * s, gm * s - bm * c
            P, Q = gs * vu * vu + vu * vv * A, -bs * vu * vu + vu * vv * C
            dP = [-vu * vv * C, vu * vv * C, 2 * gs * vu + vv * A, vu * A]
            dQ = [vu * vv * A, -vu * vv * A, -2 * bs * vu + vv * C, vu * C]
            hP = {(0, 0): -vu * vv * A, (1, 0): vu * vv * A, (1, 1): -vu * vv * A,
                  (2, 0): -vv * C, (2, 1): vv * C, (3, 0): -vu * C, (3, 1): vu * C,
                  (2, 2): 2 * gs + 0 * A, (3, 2): A}
            hQ = {(0, 0): -vu * vv * C, (1, 0): vu * vv * C, (1, 1): -vu * vv * C,
                  (2, 0): vv * A, (2, 1): -vv * A, (3, 0): vu * A, (3, 1): -vu * A,
                  (2, 2): -2 * bs + 0 * A, (3, 2): C}
        else:
            eu, ev, fu, fv = x[:, u], x[:, v], x[:, nb + u], x[:, nb + v]
            a, b, w = eu * ev + fu * fv, fu * ev - eu * fv, eu * eu + fu * fu
            one = torch.ones_like(eu)
            P, Q = gs * w + gm * a + bm * b, -bs * w + gm * b - bm * a
            dP = [2 * gs * eu + gm * ev - bm * fv, gm * eu + bm * fu,
                  2 * gs * fu + gm * fv + bm * ev, gm * fu - bm * eu]
            dQ = [-2 * bs * eu - gm * fv - bm * ev, gm * fu - bm * eu,
                  -2 * bs * fu + gm * ev - bm * fv, -gm * eu - bm * fu]
            hP = {(0, 0): 2 * gs * one, (1, 0): gm * one, (2, 2): 2 * gs * one,
                  (3, 2): gm * one, (2, 1): bm * one, (3, 0): -bm * one}
            hQ = {(0, 0): -2 * bs * one, (1, 0): -bm * one, (2, 2): -2 * bs * one,
                  (3, 2): -bm * one, (2, 1): gm * one, (3, 0): -gm * one}
        return P, Q, dP, dQ, hP, hQ

    def evaluate(self, x, lam, mask, gen_mask, pd_scale, weight, sigma):
        """f, grad f, g | h, J values, Lagrangian Hessian values (None without lam)."""
        g, nb, nl, ng = self.g, self.g.nb, self.g.nl, self.g.ng
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
        B = x.shape[0]
        on = torch.ones(B, nl, dtype=F64, device="cuda") if mask is None else mask.to(F64)
        gon = torch.ones(B, ng, dtype=F64, device="cuda") if gen_mask is None else gen_mask.to(F64)
        sc = 1.0 if pd_scale is None else pd_scale
        w = torch.ones(B, dtype=F64, device="cuda") if weight is None else weight
        mw = g.baseMVA * x[:, 2 * nb:2 * nb + ng]
        c2, c1, c0, gb = t(g.c2), t(g.c1), t(g.c0), t(g.gbus).long()
        f = w * (gon * (c2 * mw * mw + c1 * mw + c0)).sum(1)
        grad = torch.zeros(B, g.n, dtype=F64, device="cuda")
        grad[:, 2 * nb:2 * nb + ng] = w[:, None] * gon * g.baseMVA * (2 * c2 * mw + c1)
        jt, jh, ht, flows, pe, qe = [], [], [], [], [], []
        for side, end in enumerate(self.ends):
            P, Q, dP, dQ, hP, hQ = self._end(x, end)
            u = end[0]
            jt += [on * d for d in dP] + [on * d for d in dQ]
            jh += [on * 2 * (P * p + Q * q) for p, q in zip(dP, dQ)]
            pe.append(on * P), qe.append(on * Q)
            flows.append(on * (P * P + Q * Q))
            if lam is not None:
                lp, lq = lam[:, u], lam[:, nb + u]
                mu = lam[:, 2 * nb + side * nl:2 * nb + (side + 1) * nl]
                zero = torch.zeros_like(P)
                for a in range(4):
                    for b in range(a + 1):
                        p2, q2 = hP.get((a, b), zero), hQ.get((a, b), zero)
                        ht.append(on * ((lp + 2 * mu * P) * p2 + (lq + 2 * mu * Q) * q2
                                        + 2 * mu * (dP[a] * dP[b] + dQ[a] * dQ[b])))
        uu = [self.ends[0][0], self.ends[1][0]]
        gs, bs = t(g.Gs), t(g.Bs)
        if not self.cart:
            v2 = x[:, nb:2 * nb] ** 2
            d = [torch.zeros(B, nb, dtype=F64, device="cuda"), 2 * x[:, nb:2 * nb]]
        else:
            v2 = x[:, :nb] ** 2 + x[:, nb:2 * nb] ** 2
            d = [2 * x[:, :nb], 2 * x[:, nb:2 * nb]]
        pg, qg = gon * x[:, 2 * nb:2 * nb + ng], gon * x[:, 2 * nb + ng:]
        gp = self._at_bus(pe + [-pg], uu + [gb]) + gs * v2 + t(g.Pd) * sc
        gq = self._at_bus(qe + [-qg], uu + [gb]) - bs * v2 + t(g.Qd) * sc
        gh = [gp, gq] + flows + ([v2] if self.cart else [])
        j = jt + jh + [gs * d[0], gs * d[1], -bs * d[0], -bs * d[1], -gon, -gon]
        J = self._sum(j + (d if self.cart else []), self.j_at)
        H = None
        if lam is not None:
            s2 = 2 * (lam[:, :nb] * gs - lam[:, nb:2 * nb] * bs)
            if self.cart:
                s2 = s2 + 2 * lam[:, 2 * nb + 2 * nl:]
            zero = torch.zeros_like(s2)
            cost = sigma * w[:, None] * gon * 2 * c2 * g.baseMVA ** 2
            H = self._sum(ht + [s2 if self.cart else zero, zero, s2, cost], self.h_at)
        return f, grad, torch.cat(gh, 1), J, H


def _spmv(rows, val, x, cols, m):
    out = torch.zeros(x.shape[0], m, dtype=F64, device="cuda")
    return out.index_add_(1, rows, val * x[:, cols])


def _solve_blocks(case, blocks, rhs):
    """Solves the block system on the bus graph (blocks {(u, v): [B, k, k]}, rhs [nb, B, k]) by
    block elimination on a minimum-degree order; the rest, once it is one clique, by a dense LU."""
    order, nbrs = _min_degree(case)
    nb, (B, k) = len(order), rhs.shape[1:]
    place = {}
    for u, v in blocks:
        place.setdefault((u, v), len(place))
    stop = nb
    for i, (b, ring) in enumerate(zip(order, nbrs)):
        if len(ring) == nb - i - 1:
            stop = i
            break
        for u in ring:
            for v in ring:
                place.setdefault((u, v), len(place))
    rest = order[stop:]
    for u in rest:
        for v in rest:
            place.setdefault((u, v), len(place))
    S = torch.zeros(len(place), B, k, k, dtype=F64, device="cuda")
    for uv, a in blocks.items():
        S[place[uv]] = a
    t = lambda a: torch.tensor(a, device="cuda")
    y, done = rhs.clone(), []
    for b, ring in zip(order[:stop], nbrs[:stop]):
        inv = torch.linalg.inv_ex(S[place[b, b]])[0]
        if ring:
            col, row = t([place[u, b] for u in ring]), t([place[b, u] for u in ring])
            both, at = t([place[u, v] for u in ring for v in ring]), t(ring)
            F = S[col] @ inv
            S[both] -= (F[:, None] @ S[row][None]).reshape(-1, B, k, k)
            y[at] -= (F @ y[b][None, :, :, None])[..., 0]
            done.append((b, inv, row, at))
        else:
            done.append((b, inv, None, None))
    if rest:
        r = len(rest)
        full = S[t([place[u, v] for u in rest for v in rest])].reshape(r, r, B, k, k)
        full = full.permute(2, 0, 3, 1, 4).reshape(B, r * k, r * k)
        right = y[t(rest)].permute(1, 0, 2).reshape(B, r * k, 1)
        y[t(rest)] = torch.linalg.solve(full, right).reshape(B, r, k).permute(1, 0, 2)
    for b, inv, row, at in reversed(done):
        v = y[b]
        if row is not None:
            v = v - (S[row] @ y[at][..., None])[..., 0].sum(0)
        y[b] = (inv @ v[..., None])[..., 0]
    return y


def _dense_entries(rows, cols, val, pick_r, pick_c, n):
    """{(u, v): ...}-style lookup of a sparse matrix's values by row and column."""
    key = {int(r) * n + int(c): i for i, (r, c) in enumerate(zip(rows.tolist(), cols.tolist()))}
    at = [key.get(r * n + c, -1) for r, c in zip(pick_r, pick_c)]
    at = torch.tensor(at, device="cuda")
    return torch.where(at >= 0, val[:, at.clamp(min=0)], torch.zeros((), dtype=F64, device="cuda"))


def _bus_pairs(g):
    pairs = {(u, u) for u in range(g.nb)}
    for a, c in zip(g.f.tolist(), g.t.tolist()):
        pairs |= {(a, c), (c, a)}
    return sorted(pairs)


def _exact_kkt(case, seed):
    s, g = _kkt_inputs(case, seed), grid_of(case)
    M = Model(g, False)
    J, H, dx, dc, rhs = s["jval"], s["hval"], s["dx"], s["dc"], s["rhs"]
    nb, nl, ng, n, m = g.nb, g.nl, g.ng, g.n, g.m
    rx, rc = rhs[:, :n].clone(), rhs[:, n:].clone()
    # flow rows: lambda = (j dx - r) / dc; their part j j' / dc joins the Hessian
    gb = torch.as_tensor(g.gbus, device="cuda").long()
    pairs = _bus_pairs(g)
    at = {p: i for i, p in enumerate(pairs)}
    A = torch.zeros(len(pairs), case["B"], 4, 4, dtype=F64, device="cuda")
    U, V = [p[0] for p in pairs], [p[1] for p in pairs]
    for a in range(2):
        for c in range(2):
            i, j = [a * nb + u for u in U], [c * nb + v for v in V]
            lo = _dense_entries(M.h_row, M.h_col, H, [max(p) for p in zip(i, j)],
                                [min(p) for p in zip(i, j)], n)
            A[:, :, a, c] = lo.T
            A[:, :, 2 + a, c] = _dense_entries(M.j_row, M.j_col, J, i, j, n).T
            A[:, :, c, 2 + a] = _dense_entries(M.j_row, M.j_col, J, [a * nb + v for v in V],
                                               [c * nb + u for u in U], n).T
    own = torch.tensor([at[u, u] for u in range(nb)], device="cuda")
    for a in range(2):
        A[own, :, a, a] += dx[:, a * nb:(a + 1) * nb].T
        A[own, :, 2 + a, 2 + a] -= dc[:, a * nb:(a + 1) * nb].T
    f, to = g.f.tolist(), g.t.tolist()
    flow = []
    for side in range(2):
        row = [2 * nb + side * nl + l for l in range(nl)]
        d = dc[:, 2 * nb + side * nl:2 * nb + (side + 1) * nl]
        r = rc[:, 2 * nb + side * nl:2 * nb + (side + 1) * nl]
        j = {}
        for name, bus in (("f", f), ("t", to)):
            for a in range(2):
                j[name, a] = _dense_entries(M.j_row, M.j_col, J, row, [a * nb + b for b in bus], n)
        flow.append((j, d, r))
        for x1, b1 in (("f", f), ("t", to)):
            for x2, b2 in (("f", f), ("t", to)):
                where = torch.tensor([at[p] for p in zip(b1, b2)], device="cuda")
                for a in range(2):
                    for c in range(2):
                        A[:, :, a, c].index_add_(0, where, (j[x1, a] * j[x2, c] / d).T)
            for a in range(2):
                rx.index_add_(1, torch.tensor([a * nb + b for b in b1], device="cuda"),
                              j[x1, a] * r / d)
    # generators: Pg and Qg touch only their bus's balances
    gens = []
    for q in range(2):
        k = 2 * nb + q * ng
        aj = _dense_entries(M.j_row, M.j_col, J, [q * nb + b for b in g.gbus.tolist()],
                            list(range(k, k + ng)), n)
        piv = dx[:, k:k + ng]
        if q == 0:
            piv = piv + _dense_entries(M.h_row, M.h_col, H, list(range(k, k + ng)),
                                       list(range(k, k + ng)), n)
        A[:, :, 2 + q, 2 + q].index_add_(0, own[gb], -(aj * aj / piv).T)
        rc.index_add_(1, q * nb + gb, -aj * rx[:, k:k + ng] / piv)
        gens.append((k, aj, piv))
    right = torch.stack([rx[:, :nb], rx[:, nb:2 * nb], rc[:, :nb], rc[:, nb:2 * nb]], -1)
    y = _solve_blocks(case, {p: A[i] for i, p in enumerate(pairs)}, right.permute(1, 0, 2))
    sol = torch.empty_like(rhs)
    for a in range(2):
        sol[:, a * nb:(a + 1) * nb] = y[:, :, a].T
        sol[:, n + a * nb:n + (a + 1) * nb] = y[:, :, 2 + a].T
    for q, (k, aj, piv) in enumerate(gens):
        sol[:, k:k + ng] = (rx[:, k:k + ng] - aj * y[gb, :, 2 + q].T) / piv
    ff, tt = torch.tensor(f, device="cuda"), torch.tensor(to, device="cuda")
    for side, (j, d, r) in enumerate(flow):
        v = sum(j[name, a] * y[bus, :, a].T for name, bus in (("f", ff), ("t", tt))
                for a in range(2))
        sol[:, n + 2 * nb + side * nl:n + 2 * nb + (side + 1) * nl] = (v - r) / d
    return {"sol": sol, "inertia": None}


def _exact_pflow(case, seed):
    g = grid_of(case)
    x, types, scale = _pflow_inputs(case, seed)
    x = _cuda(x)
    M, nb = Model(g, False), g.nb
    _, _, gh, J, _ = M.evaluate(x, None, None, None, _cuda(scale), None, 1.0)
    free = np.stack([types != 3, types == 1], 1)   # Va (P rows) and Vm (Q rows) of each bus
    live = _cuda(free.astype(np.float64))
    gpf = torch.stack([gh[:, :nb], gh[:, nb:2 * nb]], -1) * live
    pairs = _bus_pairs(g)
    U, V = [p[0] for p in pairs], [p[1] for p in pairs]
    A = torch.zeros(len(pairs), case["B"], 2, 2, dtype=F64, device="cuda")
    for a in range(2):
        for c in range(2):
            e = _dense_entries(M.j_row, M.j_col, J, [a * nb + u for u in U],
                               [c * nb + v for v in V], g.n)
            A[:, :, a, c] = (e * live[U, a] * live[V, c]).T
    for i, (u, v) in enumerate(pairs):
        if u == v:
            for a in range(2):
                if not free[u, a]:
                    A[i, :, a, a] = 1.0
    d = _solve_blocks(case, {p: A[i] for i, p in enumerate(pairs)}, -gpf.permute(1, 0, 2))
    new = x.clone()
    for a in range(2):
        new[:, a * nb:(a + 1) * nb] += d[:, :, a].T
    return {"x": new, "mismatch": gpf.abs().amax((1, 2))}


def _exact_rows(case, seed):
    g, B = grid_of(case), case["B"]
    r = _rows_inputs(case, seed)
    at = r["row"].astype(np.int64) * g.nb + r["bus"]
    sz = r["sign"] * r["z"]
    gh = r["gh"].copy()
    np.add.at(gh.T, at, sz.T)
    parent = synth.coupling_parents(case["tie"], B)
    pg, tied = r["x"][:, 2 * g.nb:2 * g.nb + g.ng], parent >= 0
    rows, ct = np.zeros((B, g.ng)), np.zeros((B, g.ng))
    rows[tied] = pg[tied] - pg[parent[tied]]
    ct[tied] = r["nu"][tied]
    np.add.at(ct, parent[tied], -r["nu"][tied])
    return {"gh": gh, "f": r["weight"] * (r["cost"] * r["z"]).sum(1),
            "grad_z": r["weight"][:, None] * r["cost"], "jtv_z": r["sign"] * r["v"][:, at],
            "r": rows, "ct_nu": ct}


def exact(case, seed):
    kind = case["kind"]
    if kind == "kkt":
        return _exact_kkt(case, seed)
    if kind == "pflow":
        return _exact_pflow(case, seed)
    if kind == "rows":
        return _exact_rows(case, seed)
    g, b = grid_of(case), _batch(case, seed)
    M = Model(g, kind == "cart")
    f, grad, gh, J, H = M.evaluate(_cuda(b["x"]), _cuda(b["lam"]), _cuda(b["mask"]),
                                   _cuda(b["gen_mask"]), _cuda(b["pd_scale"]),
                                   _cuda(b["weight"]), 1.0)
    if kind == "adjoint":
        u, v = _randn(seed, case["B"], g.n), _randn(seed + 1, case["B"], g.m)
        r, c, hr, hc = M.j_row, M.j_col, M.h_row, M.h_col
        off = hr != hc
        hu = _spmv(hr, H, u, hc, g.n) + _spmv(hc[off], H[:, off], u, hr[off], g.n)
        return {"ju": _spmv(r, J, u, c, g.m), "jtv": _spmv(c, J, v, r, g.n), "hu": hu}
    if case["want"] == "trial":
        return {"f": f, "gh": gh}
    return {"f": f, "grad": grad, "gh": gh, "jval": J, "hval": H}
