"""The performance cases: what users of the library have it do, at the sizes
they do it, each through the public entry points of the ctypes binding.

A user runs an interior-point method.  The pattern of its grid is analysed
once; every iteration brings new values (barrier diagonals, the coupling
diagonal, a right-hand side), so a pass is the numeric work of one iteration:

    step    kkt_factor, then kkt_solve (refined), on one handle; with "host"
            the values come from and the solution goes to pinned host memory
    solve   kkt_solve alone on a factored handle: corrector and second-order
            right-hand sides, `nrhs` of them in one call
    batch   kkt_batch_factor_solve of several independent grids at once
    slack   the slack elimination before the solve and the recovery after it

Three couplings: "adjacent" (the storage states of neighbouring periods, a
banded S), "paper" (the cumulative energy constraints, S of repeated blocks:
s = 2) and "scopf" (nominal grid and line outages, a dense C and S).  s is
kkt_options.structured_s (0 dense S, 1 its row envelope, 2 repeated blocks).

The barrier diagonals are log-uniform over 10^-bar .. 10^bar and the
tolerance of the refinement is tight, as in an interior-point iterate whose
step is wanted to full accuracy: at the late-iteration range 1e-8 .. 1e8 the
condition of K leaves a few digits of the solution at most, and two correct
solvers agree on little more than the residual.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from gen import GridSpec, make_problem, make_scopf
from paper_1907_05420_gb300 import binding as B


def _case(name, kind, buses, lines, gens, stor, per, *, coupling="adjacent", prec="fp64", s=0, gmres=0, tol=1e-16,
          nrhs=1, host=False, bar=3.0, limits=0, count=1):
    c = {"kind": kind, "buses": buses, "lines": lines, "gens": gens, "stor": stor, "per": per, "coupling": coupling,
         "prec": prec, "s": s, "gmres": gmres, "tol": tol, "nrhs": nrhs, "host": host, "bar": bar, "limits": limits,
         "count": count}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system a user solves, thousands of times in a row: launches and latency
        _case("step 30 bus 24 per fp64", "step", 30, 40, 6, 3, 24),
        # its corrector right-hand side
        _case("solve 30 bus 24 per fp64", "solve", 30, 40, 6, 3, 24),
        # a regional grid of odd size, every factor in FP64, S by its envelope
        _case("step 301 bus 48 per fp64", "step", 301, 391, 45, 23, 48, s=1),
        # the same kind of grid larger, emulated FP64, values in host memory (an IPM written for the CPU)
        _case("step 1021 bus 24 per f64emu host", "step", 1021, 1327, 153, 77, 24, prec="f64emu", host=True),
        # a national grid over four days in hours: plain FP64, S by its envelope
        _case("step 2383 bus 96 per fp64", "step", 2383, 2900, 327, 100, 96, s=1),
        # the mixed-precision path on it: TF32 factor of the dense S, GMRES refinement
        _case("step 2383 bus 96 per tf32", "step", 2383, 2900, 327, 100, 96, prec="tf32", gmres=1),
        # several right-hand sides on its factors
        _case("solve 2383 bus 96 per fp64", "solve", 2383, 2900, 327, 100, 96, s=1, nrhs=4),
        # the cumulative coupling, whose S is dense but made of repeated blocks
        _case("step 2383 bus 96 per cumulative", "step", 2383, 2900, 327, 100, 96, coupling="paper", prec="f64emu",
              s=2),
        # security-constrained OPF: 16 line outages, dense S
        _case("step 1021 bus scopf 16", "step", 1021, 1327, 153, 0, 17, coupling="scopf", prec="f64emu"),
        # a continental grid over a day: the largest
        _case("step 9241 bus 24 per f64emu", "step", 9241, 16049, 1445, 400, 24, prec="f64emu"),
        # uneven grids from several users at once
        _case("batch 12 grids fp64", "batch", 240, 312, 36, 18, 24, s=1, count=12),
        # slack elimination and recovery around the solve, a flow limit on every line
        _case("slack 2383 bus 96 per", "slack", 2383, 2900, 327, 100, 96, limits=2900),
    ]


def draw(rng):
    """Grids of 30 to 2,383 buses (log-uniform) with the line, generator and
    storage densities of the listed ones, 4 to 96 periods, every kind."""
    buses = round(math.exp(rng.uniform(math.log(30), math.log(2384))))
    lines = buses + round(buses * rng.uniform(0.21, 0.33))
    gens = max(2, round(buses * rng.uniform(0.13, 0.2)))
    stor = max(1, round(buses * rng.uniform(0.04, 0.10)))
    per = rng.randint(4, 96)
    kind = rng.choice(["step", "step", "step", "step", "solve", "slack", "batch"])
    prec = rng.choice(["fp64", "f64emu", "tf32"])
    if kind == "batch":
        buses = min(buses, 600)
        return _case(None, kind, buses, round(1.3 * buses), max(2, round(0.15 * buses)),
                     max(1, round(0.07 * buses)), rng.choice([12, 24, 48]), s=1, count=rng.randint(2, 12))
    if kind == "slack":
        return _case(None, kind, buses, lines, gens, stor, per, limits=rng.randint(1, lines))
    coupling = rng.choice(["adjacent", "adjacent", "paper", "scopf"])
    if coupling == "scopf":
        buses = min(buses, 1021)
        lines, gens = min(lines, round(1.3 * buses)), min(gens, round(0.2 * buses))
        return _case(None, kind, buses, lines, gens, 0, 1 + rng.randint(1, max(1, min(16, lines - buses))),
                     coupling="scopf", prec=prec, gmres=int(prec == "tf32"))
    if coupling == "paper":
        return _case(None, kind, buses, lines, gens, min(stor, 100), per, coupling="paper",
                     prec=rng.choice(["fp64", "f64emu"]), s=2)
    stor = min(stor, max(1, 9600 // per))
    s = 1 if prec == "fp64" else rng.choice([0, 1])
    return _case(None, kind, buses, lines, gens, stor, per, prec=prec, s=s, gmres=int(prec == "tf32"),
                 nrhs=rng.choice([1, 2, 4]) if kind == "solve" else 1, host=kind == "step" and rng.random() < 0.25)


# ---- inputs ----

@functools.lru_cache(maxsize=16)
def _pattern(coupling, buses, lines, gens, stor, per, limits):
    """The grid and its coupling with a unit barrier: the pattern and the values that no iteration changes."""
    spec = GridSpec(buses, lines, gens, max(stor, 1), per, 1.0, 1.0, 1907 + buses)
    if coupling == "scopf":
        return make_scopf(spec, per - 1)
    return make_problem(spec, coupling=coupling, flow_limits=limits)


def _members(case):
    """The (coupling, sizes) of every system of the case; a batch takes grids
    between half and twice its size."""
    n = case["count"]
    out = []
    for i in range(n):
        f = 1.0 if n == 1 else 2.0 ** (2.0 * i / (n - 1) - 1.0)
        nb = max(8, round(case["buses"] * f))
        if n == 1:
            sizes = (case["buses"], case["lines"], case["gens"], case["stor"])
        else:
            sizes = (nb, round(1.3 * nb), max(2, round(0.15 * nb)), max(1, round(0.07 * nb)))
        out.append((case["coupling"], *sizes, case["per"], case["limits"]))
    return out


def _log_uniform(g, lo, hi, *shape):
    return 10.0 ** (lo + (hi - lo) * torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda"))


def _values(p, case, g):
    """One iteration's values (a, b, c, rhs) on the device."""
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to("cuda")  # noqa: E731
    a = up(p.a_vals).reshape(p.N, -1).clone()
    pos = up(p.bar_pos)
    bar = _log_uniform(g, -case["bar"], case["bar"], p.N, len(p.bar_pos))
    a[:, pos] += bar - 1.0
    b, c = up(p.b_vals), up(p.c_vals).clone()
    if case["coupling"] == "adjacent":
        c = _log_uniform(g, -case["bar"], case["bar"], p.nC)
    elif case["coupling"] == "scopf":
        c.view(p.nC, p.nC).diagonal().add_(_log_uniform(g, -case["bar"], case["bar"], p.nC) - 1.0)
    rhs = torch.randn(case["nrhs"], p.nK, generator=g, dtype=torch.float64, device="cuda")
    return a, b, c, rhs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


class _System:
    """One analysed grid with an iteration's values; frees its handle with itself."""

    def __init__(self, p, case, g):
        self.p = p
        opts = {"structured_s": case["s"], "refine_mode": case["gmres"], "refine_tol": case["tol"], "max_refine": 30}
        if case["coupling"] == "adjacent" and case["buses"] > 4000:
            opts["tail_ratio"] = 1.25  # what the autotuner finds for grids of this size
        self.solver = B.KKTSolver(p, case["prec"], **opts)
        self.h = self.solver.h
        vals = _values(p, case, g)
        if case["host"]:
            vals = tuple(v.cpu().pin_memory().numpy() for v in vals)
            self.x = torch.empty(vals[3].shape, dtype=torch.float64).pin_memory().numpy()
        else:
            self.x = torch.empty_like(vals[3])
        self.a, self.b, self.c, self.rhs = vals


def _slack_state(p, case, g):
    nx, nd, L = p.N * p.nP + p.nC, p.N * (p.nA - p.nP), p.N * len(p.ineq_rows)
    n = lambda k: torch.randn(k, generator=g, dtype=torch.float64, device="cuda")  # noqa: E731
    x, s = _log_uniform(g, -2, 0, nx), _log_uniform(g, -2, 0, L)
    st = {"x": x, "z": x * _log_uniform(g, -case["bar"], case["bar"], nx), "s": s, "y": s * _log_uniform(g, -2, 2, L),
          "la": n(nx), "le": n(nx), "lcd": n(nd), "lb": n(L), "lf": n(L)}
    a_base = torch.from_numpy(p.a_const).to("cuda").expand(p.N, -1).contiguous()
    c_base = torch.zeros(p.nC, dtype=torch.float64, device="cuda")
    return st, a_base, c_base, n(p.nK) * _log_uniform(g, -3, 3, p.nK)


def prepare(case, seed):
    g = _generator(seed)
    ps = [_pattern(*m) for m in _members(case)]
    if case["kind"] == "slack":
        p = ps[0]
        solver = B.KKTSolver(p, case["prec"])
        st, a_base, c_base, dsol = _slack_state(p, case, g)
        e = torch.empty_like
        return {"kind": "slack", "solver": solver, "slack": B.Slack(solver.h, p.ineq_rows), "st": st, "a": a_base,
                "c": c_base, "dsol": dsol, "out": (e(a_base), e(c_base), e(dsol)),
                "rec": (e(st["s"]), e(st["x"]), e(st["s"]))}
    sys_ = [_System(p, case, g) for p in ps]
    if case["kind"] == "solve":
        B.kkt_factor(sys_[0].h, sys_[0].a, sys_[0].b, sys_[0].c)
    return {"kind": case["kind"], "sys": sys_, "nrhs": case["nrhs"]}


def run(state):
    kind = state["kind"]
    if kind == "slack":
        state["slack"].reduce(state["st"], state["a"], state["c"], *state["out"])
        state["slack"].recover(state["st"], state["dsol"], *state["rec"])
        return {"reduced": state["out"], "recovered": state["rec"]}
    if kind == "batch":
        s = state["sys"]
        B.kkt_batch_factor_solve([v.h for v in s], [v.a for v in s], [v.b for v in s], [v.c for v in s],
                                 [v.rhs for v in s], [v.x for v in s], streams=8)
        return [v.x for v in s]
    s = state["sys"][0]
    if kind == "step":
        B.kkt_factor(s.h, s.a, s.b, s.c)
    B.kkt_solve(s.h, s.rhs, s.x, state["nrhs"], allow_not_converged=True)
    return s.x


# ---- the work of a pass ----

def _system_work(m, case):
    """Bytes and operations of one system.  The factor's size follows the
    meshes of the grid (lines beyond a spanning tree, e): about 0.5 e^2 + 20 nA
    entries and 0.3 e^3 + 4500 nA operations per block for the orderings known
    for such grids; S is factored by its structure."""
    p = _pattern(*m)
    _, buses, lines, _, stor, per, _ = m
    e = lines - (buses - 1)
    nnz_l = 0.5 * e * e + 20.0 * p.nA
    if case["coupling"] == "scopf":
        s_flops, s_entries = p.nC ** 3 / 3.0, p.nC ** 2 / 2.0
    else:
        s_flops, s_entries = per * 7.0 / 3.0 * stor ** 3, per * 1.5 * stor ** 2
    values = p.N * p.nnzA + len(p.b_vals) + len(p.c_vals)
    if case["kind"] == "slack":
        L = p.N * len(p.ineq_rows)
        nx = p.N * p.nP + p.nC
        moved = 2 * values - 2 * len(p.b_vals) + 2 * p.nK + 5 * nx + p.N * (p.nA - p.nP) + 6 * L
        return 8.0 * moved, 6.0 * nx + 12.0 * L
    solve = 4.0 * case["nrhs"] * (p.N * (nnz_l + 2 * p.nnzA) + s_entries)
    if case["kind"] == "solve":
        return 8.0 * (p.N * nnz_l + s_entries + values + 2 * case["nrhs"] * p.nK), solve
    return 8.0 * (values + 2 * p.nK), p.N * (0.3 * e ** 3 + 4500.0 * p.nA) + s_flops + solve


def work(case):
    w = [_system_work(m, case) for m in _members(case)]
    return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}


# ---- the same in 64 bits, dense, by torch ----

def _exact_system(p, a, b, c, rhs):
    """x with K x = rhs: block elimination with a dense LU of every A_i, then
    two steps of refinement on the sparse K."""
    dev = a.device
    N, nA, nC = p.N, p.nA, p.nC
    rowptr, col = (torch.from_numpy(np.asarray(v, dtype=np.int64)).to(dev) for v in (p.a_rowptr, p.a_col))
    row = torch.repeat_interleave(torch.arange(nA, device=dev), rowptr.diff())
    brow, bcol = (torch.from_numpy(np.asarray(v, dtype=np.int64)).to(dev) for v in (p.b_row, p.b_col))
    bp = [int(v) for v in p.b_blockptr]
    Cm = torch.diag(c) if p.c_kind == 0 else c.view(nC, nC)
    E = torch.unique(brow)                       # the rows of A that carry B
    at = torch.zeros(nA, dtype=torch.int64, device=dev)
    at[E] = torch.arange(len(E), device=dev)
    lus, G, AE = [], [], []
    unit = torch.zeros(nA, len(E), dtype=torch.float64, device=dev)
    unit[E, torch.arange(len(E), device=dev)] = 1.0
    S = Cm.clone()
    Ms = []
    for i in range(N):
        A = torch.zeros(nA, nA, dtype=torch.float64, device=dev)
        A[row, col] = a[i]
        A[col, row] = a[i]
        lus.append(torch.linalg.lu_factor(A))
        AE.append(torch.linalg.lu_solve(*lus[i], unit))
        G.append(AE[i][E])
        q = slice(bp[i], bp[i + 1])
        used = torch.unique(bcol[q])
        M = torch.zeros(len(E), len(used), dtype=torch.float64, device=dev)
        M[at[brow[q]], torch.searchsorted(used, bcol[q])] = b[q]
        Ms.append((used, M))
        S[used[:, None], used[None, :]] -= M.T @ G[i] @ M
    slu = torch.linalg.lu_factor(S)

    def solve(r):
        rb, rg = r[:N * nA].view(N, nA), r[N * nA:].clone()
        z = [torch.linalg.lu_solve(*lus[i], rb[i][:, None])[:, 0] for i in range(N)]
        for i in range(N):
            used, M = Ms[i]
            rg[used] -= M.T @ z[i][E]
        xg = torch.linalg.lu_solve(*slu, rg[:, None])[:, 0]
        out = [z[i] - AE[i] @ (Ms[i][1] @ xg[Ms[i][0]]) for i in range(N)]
        return torch.cat(out + [xg])

    def times(x):
        xb, xg = x[:N * nA].view(N, nA), x[N * nA:]
        off = row != col
        y = torch.zeros(N, nA, dtype=torch.float64, device=dev)
        y.index_add_(1, row, a * xb[:, col])
        y.index_add_(1, col[off], a[:, off] * xb[:, row[off]])
        yg = Cm @ xg
        for i in range(N):
            q = slice(bp[i], bp[i + 1])
            y[i].index_add_(0, brow[q], b[q] * xg[bcol[q]])
            yg.index_add_(0, bcol[q], b[q] * xb[i][brow[q]])
        return torch.cat([y.reshape(-1), yg])

    out = []
    for r in rhs:
        x = solve(r)
        for _ in range(2):
            x = x + solve(r - times(x))
        out.append(x)
    return torch.stack(out)


def _exact_slack(p, st, a_base, c_base, dsol):
    """The slack elimination and its recovery, written out."""
    N, nP, nA, nC = p.N, p.nP, p.nA, p.nC
    dev = a_base.device
    rowptr, col = (torch.from_numpy(np.asarray(v, dtype=np.int64)).to(dev) for v in (p.a_rowptr, p.a_col))
    row = torch.repeat_interleave(torch.arange(nA, device=dev), rowptr.diff())
    diag = torch.nonzero(row == col)[:, 0]       # one per row, in row order
    ineq = torch.from_numpy(np.asarray(p.ineq_rows, dtype=np.int64)).to(dev)
    nb = N * nP
    blocks = lambda v: v.view(N, -1)             # noqa: E731
    x, z, la, le = st["x"], st["z"], st["la"], st["le"]
    s, y, lb, lf = (blocks(st[k]) for k in ("s", "y", "lb", "lf"))
    lcd = blocks(st["lcd"])
    a = a_base.clone()
    a[:, diag[:nP]] += blocks((z / x)[:nb])
    a[:, diag[ineq]] = -(s / y)
    r = torch.empty(N, nA, dtype=torch.float64, device=dev)
    r[:, :nP] = blocks(-(la + le / x)[:nb])
    r[:, nP:] = -lcd
    r[:, ineq] = -(lcd[:, ineq - nP] + s / y * (lb + lf / s))
    rhs = torch.cat([r.reshape(-1), -(la + le / x)[nb:]])
    d = dsol[:N * nA].view(N, nA)
    dx = torch.cat([d[:, :nP].reshape(-1), dsol[N * nA:]])
    ds = s / y * (d[:, ineq] - lb - lf / s)
    dz = -(le + z * dx) / x
    dy = -(lf + y * ds) / s
    return {"reduced": (a, c_base + (z / x)[nb:], rhs), "recovered": (ds.reshape(-1), dz, dy.reshape(-1))}


def exact(case, seed):
    g = _generator(seed)
    ps = [_pattern(*m) for m in _members(case)]
    if case["kind"] == "slack":
        return _exact_slack(ps[0], *_slack_state(ps[0], case, g))
    # dense block factors: up to 4e12 operations and 20 GB
    if sum(2 / 3 * p.N * p.nA ** 3 for p in ps) > 4e12 or any(8 * p.N * p.nA ** 2 > 2e10 or p.nC > 8000 for p in ps):
        return None
    xs = [_exact_system(p, *_values(p, case, g)) for p in ps]
    if case["kind"] == "batch":
        return xs
    return xs[0]
