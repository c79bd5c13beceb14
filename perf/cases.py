"""What the framework is timed on: the calls a user of the library makes, over the sizes,
precisions and options in which they are made.

Kinds of call (a case's ``kind``):

``residual``   scylla_primal_residual_noalloc on a caller's device arrays
``solve``      a budgeted PDHG solve of one LP relaxation from the cold start
``round``      one feasibility-pump round: objective update, solve, fix-and-propagate,
               the exact feasibility test
``batch``      many LP relaxations solved together
``fanout``     K pump objectives of one LP solved together
``propagate``  bound propagation on the GPU
``create``     a new handle: upload, transpose, tiles, preconditioning

A solve's budget is one check interval of attempts: the adaptive step rule makes long
runs chaotic under rounding, so the points that two roundings of the same method reach
stay comparable only over such a budget.  The interval is the default (``n_check`` = 64),
32 in FP32-mixed solves and on integer coefficients, which diverge sooner, and 16 in pump
rounds and in the fan-out, whose tile shapes are timed when it is made and differ in
rounding.
Results of FP32-mixed solves are returned in FP32, the type their iterates have.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2307_03466_gb300 import instances as I
from paper_2307_03466_gb300 import scylla as S

CHECK = 64  # attempts between KKT checks (the default)
SHORT_CHECK = 32  # in FP32-mixed solves and those of set-cover and knapsack LPs
ROUND_CHECK = 16  # in pump rounds
FAN_CHECK = 16  # in the fan-out's solves


# --------------------------------------------------------------------- the cases ---
def listed():
    return [
        # the smallest call: the feasibility of a point on the repository's set-cover
        # workload, as a real-time caller polls it
        {"name": "residual set cover", "kind": "residual", "family": "set_cover", "m": 200, "n": 500},
        # the same on the fan-out workload's LP (5M nonzeros)
        {"name": "residual 5M", "kind": "residual", "family": "pack_cover", "m": 200_000, "n": 500_000,
         "per_col": 10},
        # the default precision on the smallest workload: pump rounds of small MIPs
        {"name": "solve set cover fp64", "kind": "solve", "family": "set_cover", "m": 200, "n": 500, "mixed": False,
         "attempts": SHORT_CHECK},
        # a mid-size LP (the batched workload's kind and a middle size of its range)
        {"name": "solve knapsack mixed", "kind": "solve", "family": "knapsack", "m": 4999, "mixed": True,
         "attempts": SHORT_CHECK},
        # the headline workload of bench.py in both precisions: 1M nonzeros, in L2
        {"name": "solve pack/cover mixed", "kind": "solve", "family": "pack_cover", "m": 50_000, "n": 100_000,
         "per_col": 10, "mixed": True, "attempts": SHORT_CHECK},
        {"name": "solve pack/cover fp64", "kind": "solve", "family": "pack_cover", "m": 50_000, "n": 100_000,
         "per_col": 10, "mixed": False, "attempts": CHECK},
        # network design: 12.8M nonzeros, short rows and 500-entry ones, out of L2
        {"name": "solve mcf mixed", "kind": "solve", "family": "mcf", "nodes": 1000, "commodities": 500, "mixed": True,
         "attempts": SHORT_CHECK},
        # a pump round on a binary MIP, default parameters
        {"name": "round binary fp64", "kind": "round", "m": 8000, "n": 20_000, "per_col": 10, "round": 3,
         "mixed": False, "attempts": ROUND_CHECK},
        # many LPs of power-law size
        {"name": "batch 64 mixed", "kind": "batch", "count": 64, "m_min": 1000, "m_max": 50_000, "mixed": True,
         "attempts": SHORT_CHECK},
        # 64 rounding targets of one LP
        {"name": "fanout 64 mixed", "kind": "fanout", "m": 80_000, "n": 200_000, "per_col": 10, "K": 64,
         "mixed": True, "attempts": FAN_CHECK},
        # propagation of the headline workload's bounds
        {"name": "propagate pack/cover", "kind": "propagate", "family": "pack_cover", "m": 50_000, "n": 100_000,
         "per_col": 10},
        # a new handle for the headline workload
        {"name": "create pack/cover mixed", "kind": "create", "family": "pack_cover", "m": 50_000, "n": 100_000,
         "per_col": 10, "mixed": True},
    ]


def draw(rng):
    def size(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def instance(families, top):
        f = rng.choice(families)
        if f == "set_cover":
            return {"family": f, "m": size(60, 400), "n": size(300, 1200)}
        if f == "knapsack":
            return {"family": f, "m": size(300, min(50_000, top // 16))}
        if f == "mcf":
            k = size(20, 300)
            return {"family": f, "nodes": size(50, max(60, min(1000, top // (26 * k)))), "commodities": k}
        per_col = rng.randint(3, 12)
        m = size(500, max(1000, top // (2 * per_col)))
        return {"family": f, "m": m, "n": int(m * rng.uniform(1.3, 2.5)), "per_col": per_col}

    kind = rng.choice(["residual", "solve", "solve", "solve", "round", "batch", "fanout", "propagate", "create"])
    mixed = rng.random() < 0.5
    if kind == "residual":
        return {"kind": kind, **instance(["set_cover", "knapsack", "pack_cover", "mcf"], 4_000_000)}
    if kind == "solve":
        c = instance(["set_cover", "knapsack", "pack_cover", "pack_cover", "mcf"], 6_000_000)
        short = mixed or c["family"] in ("set_cover", "knapsack")
        return {"kind": kind, **c, "mixed": mixed, "attempts": SHORT_CHECK if short else CHECK}
    if kind == "round":
        m = size(500, 20_000)
        return {"kind": kind, "m": m, "n": int(m * rng.uniform(1.5, 3.0)), "per_col": rng.randint(4, 11),
                "round": rng.randint(1, 8), "mixed": mixed, "attempts": ROUND_CHECK}
    if kind == "batch":
        a = size(300, 2000)
        return {"kind": kind, "count": rng.randint(5, 63), "m_min": a, "m_max": a * rng.randint(2, 20), "mixed": mixed,
                "attempts": SHORT_CHECK}
    if kind == "fanout":
        m = size(2000, 60_000)
        return {"kind": kind, "m": m, "n": int(m * rng.uniform(1.5, 2.5)), "per_col": rng.randint(5, 10),
                "K": rng.choice([3, 8, 16, 17, 31, 48, 64]), "mixed": True, "attempts": FAN_CHECK}
    families = ["knapsack", "pack_cover"] if kind == "propagate" else ["knapsack", "pack_cover", "mcf"]
    return {"kind": kind, **instance(families, 2_000_000), "mixed": mixed}


def _instance(case, seed):
    f = case["family"]
    if f == "set_cover":
        return I.set_cover(case["m"], case["n"], seed=seed)
    if f == "knapsack":
        return I.knapsack_cover(case["m"], seed=seed)
    if f == "mcf":
        # one network of each size; the costs change from seed to seed
        inst = I.mcf(nodes=case["nodes"], commodities=case["commodities"])
        inst.c = inst.c * np.random.default_rng(seed).uniform(0.5, 1.5, inst.n)
        return inst
    return I.packing_covering(case["m"], case["n"], case["per_col"], seed=seed)


def _instances(case, seed):
    sizes = I.power_law_sizes(case["count"], case["m_min"], case["m_max"])
    return [I.knapsack_cover(int(m), seed=seed * 1000 + b) for b, m in enumerate(sizes)]


def _point(inst, seed):
    """A point as a heuristic has it: most entries at their lower bound."""
    rng = np.random.default_rng(seed + 1)
    return np.where(rng.random(inst.n) < 0.7, 0.0, rng.uniform(0.0, 1.0, inst.n)) * np.minimum(inst.u, 100.0)


def _binary(case, seed):
    return I.fanout_base(case["m"], case["n"], case["per_col"], seed=seed)


def _targets(inst, K, seed):
    base = (np.random.default_rng(seed).random(inst.n) < 0.5) * inst.is_int.astype(np.float64)
    return I.fanout_targets(inst, base, K, seed=seed + 1)


def _params(case, **kw):
    return S.default_params(precision=S.PREC_MIXED if case.get("mixed") else S.PREC_FP64,
                            n_check=case.get("attempts", CHECK), **kw)


# ---------------------------------------------------------------- prepare and run ---
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "residual":
        inst = _instance(case, seed)
        dev = "cuda"
        for k, a in (("rowptr", inst.rowptr), ("cols", inst.cols), ("vals", inst.vals), ("x", _point(inst, seed)),
                     ("lo", inst.lo), ("hi", inst.hi)):
            st[k] = torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        st["m"] = inst.m
        st["out"] = torch.zeros(2, dtype=torch.float64, device=dev)
    elif kind == "solve":
        st["lp"] = S.LP.from_instance(_instance(case, seed), _params(case, aux_general_integers=0))
    elif kind == "round":
        inst = _binary(case, seed)
        st["lp"] = S.LP.from_instance(inst, _params(case))
        st["xhat"] = np.ascontiguousarray(_targets(inst, 1, seed)[:, 0])
    elif kind == "batch":
        insts = _instances(case, seed)
        st["batch"] = S.Batch(insts, _params(case))
        st["x"] = np.empty(sum(i.n for i in insts), dtype=_float(case))
        st["y"] = np.empty(sum(i.m for i in insts), dtype=_float(case))
    elif kind == "fanout":
        inst = _binary(case, seed)
        st["lp"] = S.LP.from_instance(inst, _params(case, aux_general_integers=0))
        st["fan"] = S.Fanout(st["lp"], _targets(inst, case["K"], seed))
        st["x"] = np.empty((case["K"], inst.n), dtype=_float(case))
    elif kind == "propagate":
        inst = _instance(case, seed)
        st["lp"] = S.LP.from_instance(inst, _params(case, aux_general_integers=0))
        st["l"], st["u"] = inst.l, inst.u
    else:
        st["inst"] = _instance(case, seed)
    return st


def _float(case):
    return np.float32 if case.get("mixed") else np.float64


def _result(r, f):
    out = {k: f(getattr(r, k)) for k in ("eps_p", "eps_d", "eps_g", "eta", "omega")}
    out["objectives"] = np.array([r.pobj, r.dobj], dtype=f)
    out["iterations"] = int(r.iterations)
    return out


def _results(rs, f):
    out = {k: np.array([getattr(r, k) for r in rs], dtype=f)
           for k in ("eps_p", "eps_d", "eps_g", "eta", "omega")}
    out["objectives"] = np.array([[r.pobj, r.dobj] for r in rs], dtype=f)
    out["iterations"] = np.array([r.iterations for r in rs], dtype=np.int64)
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    f = _float(case)
    if kind == "residual":
        S.primal_residual_noalloc(state["m"], state["rowptr"].data_ptr(), state["cols"].data_ptr(),
                                  state["vals"].data_ptr(), state["x"].data_ptr(), state["lo"].data_ptr(),
                                  state["hi"].data_ptr(), state["out"].data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if kind == "solve":
        lp = state["lp"]
        lp.reset_state()
        r = lp.pdhg_solve(0.0, case["attempts"])
        return {"x": lp.primal().astype(f), "y": lp.dual().astype(f), **_result(r, f)}
    if kind == "round":
        lp = state["lp"]
        lp.reset_state()
        lp.set_objective(state["xhat"], case["round"])
        r = lp.pdhg_solve(0.0, case["attempts"])
        x = lp.primal()
        xhat = lp.fix_and_propagate(x)[0]
        ok = lp.check_feasible(xhat)
        return {"x": x.astype(f), "xhat": xhat.astype(f), "feasible": ok, **_result(r, f)}
    if kind == "batch":
        b = state["batch"]
        b.reset_state()
        rs, _ = b.solve(0.0, case["attempts"])
        x, y, p, q = state["x"], state["y"], 0, 0
        for k, (m, n) in enumerate(b.sizes):
            x[p:p + n], y[q:q + m] = b.primal(k), b.dual(k)
            p, q = p + n, q + m
        return {"x": x, "y": y, **_results(rs, f)}
    if kind == "fanout":
        fan = state["fan"]
        fan.reset_state()
        rs, _ = fan.solve(0.0, case["attempts"])
        for k in range(fan.K):
            state["x"][k] = fan.primal(k)
        return {"x": state["x"], **_results(rs, f)}
    if kind == "propagate":
        dl, du, ignored, rounds, conflicts = state["lp"].propagate(state["l"], state["u"])
        return {"dom_lo": dl, "dom_hi": du, "ignored": ignored, "rounds": rounds, "conflicts": conflicts}
    lp = S.LP.from_instance(state["inst"], _params(case, aux_general_integers=0))
    R, C = lp.scaling()
    _, _, eta, omega = lp.get_state()
    lp.close()
    return {"R": R, "C": C, "eta": np.float64(eta), "omega": np.float64(omega)}


# ---------------------------------------------------------------------------- work ---
def _sizes(case):
    """(m, n, nnz) of a case's LP (a set cover's and an mcf's as expected values)."""
    f = case.get("family", "pack_cover")
    if f == "set_cover":
        return case["m"], case["n"], int(5.5 * case["n"])
    if f == "knapsack":
        return case["m"], 2 * case["m"], 16 * case["m"]
    if f == "mcf":
        arcs, k = 8 * case["nodes"], case["commodities"]
        f_cols, z = arcs * k, arcs * k // 10
        return case["nodes"] * k + arcs + z, f_cols + arcs + z, 3 * f_cols + arcs + 2 * z
    return case["m"], case["n"], case["per_col"] * case["n"]


def _solve_work(m, n, nnz, attempts, s, K=1):
    """Bytes and operations of `attempts` PDHG attempts and two checks: per attempt one
    pass over A and one over its transpose (values of s bytes, 4-byte indices), x, y,
    their averages read and written, A x written, c and the bounds read; a check reads
    the matrix in FP64 once each way."""
    per = 2 * nnz * (4 + s) + 4 * (m + n) + K * s * (7 * n + 8 * m)
    check = 2 * nnz * 12 + K * 8 * (6 * n + 6 * m)
    return {"bytes": attempts * per + 2 * check, "flops": K * (attempts * (4 * nnz + 12 * (m + n)) + 2 * 8 * nnz)}


def work(case):
    kind = case["kind"]
    s = 4 if case.get("mixed") else 8
    if kind == "batch":
        a, b = case["m_min"], case["m_max"]
        m = int(case["count"] * math.log(b / a) * a * b / (b - a))  # mean of the m^-2 law
        return _solve_work(m, 2 * m, 16 * m, case["attempts"], s)
    m, n, nnz = _sizes(case)
    if kind == "residual":
        return {"bytes": 12 * nnz + 8 * (m + 1) + 16 * m + 8 * n + 16, "flops": 2 * nnz + 6 * m}
    if kind == "solve":
        return _solve_work(m, n, nnz, case["attempts"], s)
    if kind == "round":
        w = _solve_work(m, n, nnz, case["attempts"], s)
        # the host copies of the matrix and its transpose, read once by the propagation
        return {"bytes": w["bytes"] + 24 * nnz + 64 * (m + n), "flops": w["flops"] + 8 * nnz}
    if kind == "fanout":
        return _solve_work(m, n, nnz, case["attempts"], s, case["K"])
    if kind == "propagate":
        return {"bytes": 24 * nnz + 32 * n + 24 * m, "flops": 8 * nnz}
    # create: A in, its transpose, eleven preconditioning passes over both, the scaled
    # values out (and their FP32 copies)
    return {"bytes": 12 * nnz + 24 * nnz + 11 * 24 * nnz + 2 * (12 + 2 * (8 - s)) * nnz + 8 * 12 * (m + n),
            "flops": 11 * 6 * nnz}


# --------------------------------------------------------------------------- exact ---
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Lp:
    """An LP relaxation in 64 bits: A and its transpose as sparse tensors, the diagonal
    scaling (10 Ruiz passes, then Pock-Chambolle with alpha = 1), the scaled vectors."""

    def __init__(self, inst, c=None):
        d = _dev()
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(d)  # noqa: E731
        self.m, self.n = inst.m, inst.n
        rows = torch.from_numpy(np.repeat(np.arange(inst.m), np.diff(inst.rowptr))).to(d)
        cols = torch.from_numpy(inst.cols.astype(np.int64)).to(d)
        a = t(inst.vals)
        self.lo, self.hi, self.l, self.u = t(inst.lo), t(inst.hi), t(inst.l), t(inst.u)
        self.c = t(inst.c) if c is None else c
        R = torch.ones(self.m, dtype=torch.float64, device=d)
        C = torch.ones(self.n, dtype=torch.float64, device=d)

        def over(x, idx, count, how):
            return torch.zeros(count, dtype=torch.float64, device=d).scatter_reduce_(0, idx, x, how)

        def step(how):
            s = a.abs() * R[rows] * C[cols]
            r, q = over(s, rows, self.m, how), over(s, cols, self.n, how)
            one = torch.ones((), dtype=torch.float64, device=d)
            return R / torch.where(r > 0, r.sqrt(), one), C / torch.where(q > 0, q.sqrt(), one)

        for _ in range(10):
            R, C = step("amax")
        R, C = step("sum")
        self.R, self.C = R, C
        s = a * R[rows] * C[cols]
        self.A = torch.sparse_coo_tensor(torch.stack([rows, cols]), s, (self.m, self.n)).coalesce().to_sparse_csr()
        self.At = torch.sparse_coo_tensor(torch.stack([cols, rows]), s, (self.n, self.m)).coalesce().to_sparse_csr()
        big = torch.maximum(torch.where(self.lo.isfinite(), self.lo.abs(), 0.0),
                            torch.where(self.hi.isfinite(), self.hi.abs(), 0.0))
        self.bnorm = float(big.norm())
        q = float((big * R).norm())
        c0 = t(inst.c) * C
        self.eta0 = 1.0 / float(s.abs().max())
        self.omega0 = float(c0.norm()) / q if q > 0 and float(c0.norm()) > 0 else 1.0


def _pdhg(lp, c, offset, attempts):
    """`attempts` adaptive PDHG attempts from the cold start for the objectives in the
    columns of c (n x K), then the evaluation of the last and the averaged point; the
    one of lower relative KKT error is returned, unscaled, with its errors."""
    K = c.shape[1]
    R, C = lp.R[:, None], lp.C[:, None]
    cs = c * C
    l, u, lo, hi = lp.l[:, None] / C, lp.u[:, None] / C, lp.lo[:, None] * R, lp.hi[:, None] * R
    l, u = l.expand(-1, K), u.expand(-1, K)
    x = torch.zeros_like(cs).clamp(l, u)
    y = torch.zeros(lp.m, K, dtype=torch.float64, device=cs.device)
    ax = lp.A @ x
    eta = torch.full((K,), lp.eta0, dtype=torch.float64, device=cs.device)
    om = torch.full_like(eta, lp.omega0)
    wsum = torch.zeros_like(eta)
    xa, ya = x.clone(), y.clone()
    for k in range(1, attempts + 1):
        x2 = torch.clamp(x + (eta / om) * (lp.At @ y - cs), l, u)
        ax2 = lp.A @ x2
        sig = eta * om
        axt = 2 * ax2 - ax
        t_lo, t_hi = y + sig * (lo - axt), y + sig * (hi - axt)
        y2 = torch.where(lo.isfinite() & (t_lo > 0), t_lo, torch.where(hi.isfinite() & (t_hi < 0), t_hi, 0.0))
        dx, dy = x2 - x, y2 - y
        inter = (dy * (ax2 - ax)).sum(0).abs()
        emax = torch.where(inter > 0, (om * dx.square().sum(0) + dy.square().sum(0) / om) / (2 * inter), math.inf)
        ok = eta <= emax
        w = eta / (wsum + eta)
        nxt = torch.minimum((1 - (k + 1.0) ** -0.3) * emax, (1 + (k + 1.0) ** -0.6) * eta)
        x, y, ax = torch.where(ok, x2, x), torch.where(ok, y2, y), torch.where(ok, ax2, ax)
        xa, ya = torch.where(ok, (1 - w) * xa + w * x, xa), torch.where(ok, (1 - w) * ya + w * y, ya)
        wsum = torch.where(ok, wsum + eta, wsum)
        eta = nxt

    def evaluate(x, y):
        ax, r = (lp.A @ x) / R, (cs - lp.At @ y) / C
        o_l, o_u, o_lo, o_hi = lp.l[:, None], lp.u[:, None], lp.lo[:, None], lp.hi[:, None]
        yy, xx = y * R, x * C
        lf, uf = o_l.isfinite(), o_u.isfinite()
        lam = torch.where(lf & uf, r, torch.where(lf, r.clamp(min=0), torch.where(uf, r.clamp(max=0), 0.0)))

        def term(v, a, b):
            return (torch.where(v > 0, torch.where(a.isfinite(), a, 0.0) * v, 0.0)
                    + torch.where(v < 0, torch.where(b.isfinite(), b, 0.0) * v, 0.0)).sum(0)

        p = (c * xx).sum(0) + offset
        dd = term(yy, o_lo, o_hi) + term(lam, o_l, o_u) + offset
        ep = (ax - torch.clamp(ax, o_lo, o_hi)).norm(dim=0) / (1 + lp.bnorm)
        ed = (r - lam).norm(dim=0) / (1 + c.norm(dim=0))
        eg = (p - dd).abs() / (1 + p.abs() + dd.abs())
        return xx, yy, ep, ed, eg, p, dd

    cur, avg = evaluate(x, y), evaluate(xa, ya)
    rel = [torch.maximum(e[2], torch.maximum(e[3], e[4])) for e in (cur, avg)]
    use = (rel[1] < rel[0]) & (wsum > 0)
    out = [torch.where(use, b, a) for a, b in zip(cur, avg)]
    return out, eta, om


def _np(t):
    return t.cpu().numpy()


def _exact_solve(lp, c, offset, attempts):
    (x, y, ep, ed, eg, p, dd), eta, om = _pdhg(lp, c, offset, attempts)
    v = {"eps_p": ep, "eps_d": ed, "eps_g": eg, "eta": eta, "omega": om, "objectives": torch.stack([p, dd], dim=1)}
    return x, y, {k: _np(a) for k, a in v.items()}


def _update(inst, lp, targets, K):
    """Objectives and offsets of the pump's update of round K on binary columns."""
    d = lp.c.device
    t = torch.from_numpy(np.ascontiguousarray(targets)).to(d)
    ints = torch.from_numpy(inst.is_int.astype(bool)).to(d)[:, None]
    aK = 0.9 ** K
    s = math.sqrt(float(inst.is_int.sum())) / float(lp.c.norm())
    g = torch.where(ints, torch.where(t == lp.l[:, None], 1.0, -1.0), 0.0)
    const = torch.where(ints, torch.where(t == lp.l[:, None], -lp.l[:, None], lp.u[:, None]), 0.0).sum(0)
    return aK * s * lp.c[:, None] + (1 - aK) * g, (1 - aK) * const


def _propagate(inst):
    """The rounds of the bound propagation in 64 bits; None where rows have to be ignored
    or columns conflict (the instances have feasible points: they do not)."""
    inf, d = math.inf, _dev()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(d)  # noqa: E731
    row, j, a = t(np.repeat(np.arange(inst.m), np.diff(inst.rowptr))), t(inst.cols.astype(np.int64)), t(inst.vals)
    lo, hi, dl, du = t(inst.lo), t(inst.hi), t(inst.l).clone(), t(inst.u).clone()
    ints = t(inst.is_int.astype(bool))
    active = torch.ones(inst.m, dtype=torch.bool, device=d)
    rounds = 0

    def rowsum(v):
        return torch.zeros(inst.m, dtype=torch.float64, device=d).index_add_(0, row, v)

    while rounds < 100_000:
        rounds += 1
        pos = a > 0
        bmin, bmax = torch.where(pos, dl[j], du[j]), torch.where(pos, du[j], dl[j])
        imin, imax = bmin.isinf(), bmax.isinf()
        tmin, tmax = torch.where(imin, 0.0, a * bmin), torch.where(imax, 0.0, a * bmax)
        nmin, nmax = rowsum(imin.double()), rowsum(imax.double())
        smin, smax = rowsum(tmin), rowsum(tmax)
        if bool((active & (nmin == 0) & (smin > hi + 1e-9)).any() or (active & (nmax == 0) & (smax < lo - 1e-9)).any()):
            return None
        rmin = torch.where(nmin[row] - imin.double() == 0, smin[row] - tmin, -inf)
        rmax = torch.where(nmax[row] - imax.double() == 0, smax[row] - tmax, inf)
        up, down = (hi[row] - rmin) / a, (lo[row] - rmax) / a
        has_up, has_down = (hi[row] < inf) & (rmin > -inf), (lo[row] > -inf) & (rmax < inf)
        up, down = torch.where(has_up, up, torch.where(pos, inf, -inf)), torch.where(has_down, down,
                                                                                     torch.where(pos, -inf, inf))
        cu, cl = torch.where(pos, up, down), torch.where(pos, down, up)
        ol, ou = dl[j], du[j]
        iu, il = torch.floor(cu + 1e-6), torch.ceil(cl - 1e-6)
        bu = torch.where(ints[j], iu < ou, (cu < inf) & ((ou == inf) | (cu < ou - 1e-3 * ou.abs().clamp(min=1.0))))
        bl = torch.where(ints[j], il > ol, (cl > -inf) & ((ol == -inf) | (cl > ol + 1e-3 * ol.abs().clamp(min=1.0))))
        nu = torch.where(bu & active[row], torch.where(ints[j], iu, cu), ou)
        nl = torch.where(bl & active[row], torch.where(ints[j], il, cl), ol)
        if bool((nl > nu + 1e-9).any()):
            return None
        tl, tu = dl.scatter_reduce(0, j, nl, "amax"), du.scatter_reduce(0, j, nu, "amin")
        if bool((tl > tu + 1e-9).any()):
            return None
        moved = (tl != dl) | (tu != du)
        dl, du = tl, tu
        if not bool(moved.any()):
            break
        active = torch.zeros(inst.m, dtype=torch.bool, device=d)
        active[row[moved[j]]] = True
    return {"dom_lo": _np(dl), "dom_hi": _np(du), "ignored": None, "rounds": None, "conflicts": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "residual":
        inst = _instance(case, seed)
        x = _point(inst, seed)
        row = torch.from_numpy(np.repeat(np.arange(inst.m), np.diff(inst.rowptr)))
        ax = torch.zeros(inst.m, dtype=torch.float64).index_add_(0, row, torch.from_numpy(inst.vals * x[inst.cols]))
        lo, hi = torch.from_numpy(inst.lo), torch.from_numpy(inst.hi)
        r = float((ax - torch.clamp(ax, lo, hi)).norm())
        b = torch.maximum(torch.where(lo.isfinite(), lo.abs(), 0.0), torch.where(hi.isfinite(), hi.abs(), 0.0))
        return torch.tensor([r, r / (1.0 + float(b.norm()))], dtype=torch.float64)
    if kind == "propagate":
        return _propagate(_instance(case, seed))
    if kind == "create":
        lp = _Lp(_instance(case, seed))
        return {"R": _np(lp.R), "C": _np(lp.C), "eta": np.float64(lp.eta0), "omega": np.float64(lp.omega0)}
    if kind == "solve":
        lp = _Lp(_instance(case, seed))
        x, y, v = _exact_solve(lp, lp.c[:, None], 0.0, case["attempts"])
        return {"x": _np(x[:, 0]), "y": _np(y[:, 0]), **{k: a[0] for k, a in v.items()}, "iterations": None}
    if kind == "round":
        inst = _binary(case, seed)
        lp = _Lp(inst)
        c, off = _update(inst, lp, _targets(inst, 1, seed), case["round"])
        x, _, v = _exact_solve(lp, c, off, case["attempts"])
        # the sequential propagation takes far longer than the solve outside the library
        return {"x": _np(x[:, 0]), "xhat": None, "feasible": None, **{k: a[0] for k, a in v.items()},
                "iterations": None}
    if kind == "fanout":
        inst = _binary(case, seed)
        lp = _Lp(inst)
        c, off = _update(inst, lp, _targets(inst, case["K"], seed), 1)
        x, _, v = _exact_solve(lp, c, off, case["attempts"])
        return {"x": _np(x.T.contiguous()), **v, "iterations": None}
    xs, ys, vs = [], [], []
    for inst in _instances(case, seed):
        lp = _Lp(inst)
        x, y, v = _exact_solve(lp, lp.c[:, None], 0.0, case["attempts"])
        xs.append(_np(x[:, 0]))
        ys.append(_np(y[:, 0]))
        vs.append(v)
    return {"x": np.concatenate(xs), "y": np.concatenate(ys), **{k: np.concatenate([v[k] for v in vs]) for k in vs[0]},
            "iterations": None}
