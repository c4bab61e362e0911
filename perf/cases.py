"""Performance cases of the library: what its users have it do, end to end.

Every pass starts from host load values (or a caller's device arrays), goes
through the package's public entry points and ends with the solution in the
caller's hands.  Kinds of case:

  update     one global update on caller device arrays (opf_global_update_static)
  solve      one instance: new loads, factorization, iterations, solution
  consensus  one instance given as a consensus LP with wide, ragged blocks
  batch      many load scenarios of one feeder advanced together
  serve      a burst of requests of several feeders through the request server

A solve stops on the relative test of Sec. III-C (eps_rel > 0) or after an
iteration budget (eps_rel = 0), and a case's "iters" is its iteration count: the
budget, or about what its stopping test takes.  Results of single-precision iterations are
handed on in float32, those of double-precision iterations in float64.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2310_09410_gb300 import opf, synth

RHO, EPS_ABS = 100.0, 1e-4
PRECISION = {"fp64": opf.PREC_FP64, "mixed": opf.PREC_MIXED}


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: a control loop's allocation-free global update, with the
        # 8500-bus feeder's number of globals
        {"name": "update-63k", "kind": "update", "n": 63405},
        # the smallest solve, plain FP64 at the accuracy of the headline metric
        {"name": "solve-13-fp64", "kind": "solve", "buses": 13, "seed": 1001, "precision": "fp64", "eps_rel": 1e-8,
         "check_every": 50, "max_iter": 1000000, "iters": 3150},
        # a small feeder of the serving mix, FP32 iterations with the FP64 polish
        {"name": "solve-34-mixed", "kind": "solve", "buses": 34, "seed": 5034, "precision": "mixed", "eps_rel": 1e-8,
         "check_every": 50, "max_iter": 1000000, "iters": 12100},
        # the ordinary feeder, FP32 iterations with the FP64 polish
        {"name": "solve-123-mixed", "kind": "solve", "buses": 123, "seed": 2001, "precision": "mixed", "eps_rel": 1e-8,
         "check_every": 50, "max_iter": 1000000, "iters": 26100},
        # the same in plain FP64 at the paper's own tolerance, with the library's absolute gate (pres <= 1e-4)
        {"name": "solve-123-fp64", "kind": "solve", "buses": 123, "seed": 2001, "precision": "fp64", "eps_rel": 1e-3,
         "check_every": 50, "max_iter": 1000000, "iters": 10200},
        # the large feeder at the paper's tolerance with the paper's test (no absolute gate), both precisions
        {"name": "solve-8500-mixed", "kind": "solve", "buses": 8500, "seed": 3001, "precision": "mixed",
         "eps_rel": 1e-3, "eps_abs": 1e9, "check_every": 50, "max_iter": 1000000, "iters": 15700},
        {"name": "solve-8500-fp64", "kind": "solve", "buses": 8500, "seed": 3001, "precision": "fp64",
         "eps_rel": 1e-3, "eps_abs": 1e9, "check_every": 50, "max_iter": 1000000, "iters": 15650},
        # a caller's own consensus LP: blocks of 2 to 100 slots, too wide for a warp
        {"name": "consensus-240-mixed", "kind": "consensus", "n": 900, "blocks": 240, "widest": 100,
         "seed": 17, "precision": "mixed", "eps_rel": 0.0, "check_every": 50, "max_iter": 3000, "iters": 3050},
        # the headline batch: 1024 load scenarios to the metric's accuracy
        {"name": "batch-123x1024-mixed", "kind": "batch", "buses": 123, "seed": 2001, "instances": 1024,
         "precision": "mixed", "eps_rel": 1e-8, "check_every": 100, "max_iter": 1000000, "iters": 25940},
        # a ragged batch that does not fill the chip
        {"name": "batch-34x201-mixed", "kind": "batch", "buses": 34, "seed": 5034, "instances": 201,
         "precision": "mixed", "eps_rel": 1e-8, "check_every": 50, "max_iter": 1000000, "iters": 12100},
        # a batch in plain FP64 with an iteration budget
        {"name": "batch-123x96-fp64", "kind": "batch", "buses": 123, "seed": 2001, "instances": 96,
         "precision": "fp64", "eps_rel": 0.0, "check_every": 50, "max_iter": 2000, "iters": 2000},
        # serving: a burst of requests in the mix of the serving configuration
        {"name": "serve-45", "kind": "serve", "r13": 20, "r34": 15, "r123": 10, "eps_rel": 1e-8, "check_every": 50,
         "max_iter": 1000000, "iters": 38000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["update", "solve", "solve", "consensus", "batch", "batch", "serve"])
    if kind == "update":
        return {"kind": kind, "n": _log_int(rng, 181, 2000000)}
    if kind == "serve":
        return {"kind": kind, "r13": rng.randint(1, 20), "r34": rng.randint(1, 15), "r123": rng.randint(0, 10),
                "eps_rel": 0.0, "check_every": 50, "max_iter": 50 * rng.randint(60, 400), "iters": 0}
    case = {"kind": kind, "precision": rng.choice(["fp64", "mixed"]), "eps_rel": 0.0,
            "check_every": rng.choice([10, 50, 100])}
    budget = _log_int(rng, 500, 12000)
    if kind == "solve":
        case.update(buses=_log_int(rng, 13, 8500), seed=rng.randint(1, 10 ** 6))
    elif kind == "consensus":
        case.update(n=_log_int(rng, 60, 900), blocks=_log_int(rng, 15, 240), widest=rng.randint(8, 100),
                    seed=rng.randint(1, 10 ** 6))
        budget = min(budget, 3000)
    else:
        case.update(buses=_log_int(rng, 13, 123), seed=rng.randint(1, 10 ** 6), instances=_log_int(rng, 1, 1024))
        if case["precision"] == "fp64":     # no more work than the listed FP64 batch
            budget = max(100, min(budget, 192000 // case["instances"]))
    k = case["check_every"]
    case["max_iter"] = (budget + k - 1) // k * k
    case["iters"] = case["max_iter"]
    return case


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=8)
def _feeder(buses, seed):
    """One of the configured feeders, or a size between them with loads and DERs in proportion."""
    name = str(buses)
    if name in synth.PRESETS:
        return synth.preset_feeder(name, seed)
    share = 0.69 if buses <= 1000 else 0.14
    depth = 6 if buses < 34 else 12 if buses < 123 else 30 if buses < 1000 else 60
    single = None if buses < 100 else 0.4 if buses < 1000 else 0.7
    return synth.make_feeder(buses, max(1, int(share * buses)), max(1, buses // 12), depth_max=depth, p_single=single,
                             seed=seed)


def _scenarios(feeder, seed, count):
    """Loads of `count` scenarios: every load scaled by U[0.6, 1.2] x N(1, 0.05), [count, n_load, 3] each."""
    made = [synth.load_scenario(feeder, 1000003 * (seed % 100003) + j) for j in range(count)]
    return np.stack([m["load_a"] for m in made]), np.stack([m["load_b"] for m in made])


def _consensus(case, seed):
    """A consensus LP of random blocks (2 to `widest` slots, some rank-deficient) over boxed and some free globals;
    the structure is the case's own, the costs and right-hand sides (consistent with a point in the boxes) the seed's."""
    g = synth.random_generic(case["seed"], n_global=case["n"], n_sub=case["blocks"],
                             max_n=min(case["widest"], case["n"]), p_free=0.2)
    rng = np.random.default_rng(seed)
    point = np.clip(rng.uniform(-0.4, 0.4, case["n"]), g["lb"], g["ub"])
    subs = [dict(s, b=s["A"] @ point[s["idx"]]) for s in g["subs"]]
    return dict(g, c=rng.uniform(-1, 1, case["n"]), subs=subs)


SERVED = (("r13", 13, 5013), ("r34", 34, 5034), ("r123", 123, 5123))


def _update_arrays(case, seed):
    gen = torch.Generator().manual_seed(seed)
    n = case["n"]
    copies = torch.randint(1, 4, (n,), generator=gen)
    off = torch.zeros(n + 1, dtype=torch.int32)
    off[1:] = torch.cumsum(copies, 0)
    u = 100.0 * torch.randn(int(off[-1]), generator=gen, dtype=torch.float64)
    c = torch.where(torch.rand(n, generator=gen) < 0.1, 50.0 * torch.rand(n, generator=gen, dtype=torch.float64), 0.0)
    free = torch.rand(n, generator=gen) < 0.5
    lb = torch.where(free, -math.inf, -0.5 * torch.rand(n, generator=gen, dtype=torch.float64))
    ub = torch.where(free, math.inf, 0.5 * torch.rand(n, generator=gen, dtype=torch.float64))
    return [t.cuda() for t in (off, u, c.double(), lb.double(), ub.double())]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "update":
        off, u, c, lb, ub = _update_arrays(case, seed)
        return {"case": case, "arrays": (off, u, c, lb, ub), "x": torch.empty_like(c),
                "objective": torch.empty(1, dtype=torch.float64, device="cuda")}
    if kind == "consensus":
        g = _consensus(case, seed)
        solver = opf.Solver.from_generic(g["c"], g["lb"], g["ub"], g["subs"])
        return {"case": case, "solver": solver}
    if kind == "serve":
        server = opf.Server(rho=RHO, eps_rel=case["eps_rel"], max_iter=case["max_iter"],
                            check_every=case["check_every"], keep_solutions=True)
        models, requests = [], []
        for key, buses, feeder_seed in SERVED:
            feeder = _feeder(buses, feeder_seed)
            solver = opf.Solver.from_feeder(feeder)
            solver.precompute()
            model = server.add_model([solver], 64)
            server.set_model_shape(model, 2, 16)      # the latency-first shape of the serving configuration
            models.append(model)
            lp, lq = _scenarios(feeder, seed + buses, case[key])
            requests += [(model, lp[j], lq[j]) for j in range(case[key])]
        return {"case": case, "server": server, "models": models, "requests": requests}
    feeder = _feeder(case["buses"], case["seed"])
    solver = opf.Solver.from_feeder(feeder)
    if kind == "solve":
        lp, lq = _scenarios(feeder, seed, 1)
        return {"case": case, "solver": solver, "lp": lp[0], "lq": lq[0]}
    solver.precompute()
    n = case["instances"]
    batch = opf.Batch(solver, n)
    lp, lq = (torch.from_numpy(v).pin_memory() for v in _scenarios(feeder, seed, n))
    x = torch.empty((n, batch.n_global), dtype=torch.float64).pin_memory()
    objective = torch.empty(n, dtype=torch.float64).pin_memory()
    return {"case": case, "solver": solver, "batch": batch, "lp": lp, "lq": lq, "x": x, "objective": objective}


# ------------------------------------------------------------------- passes
def _handed_on(case, x, objective):
    kind = torch.float64 if case.get("precision") == "fp64" else torch.float32
    return {"x": torch.as_tensor(x).to(kind), "objective": torch.as_tensor(objective).to(kind)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "update":
        off, u, c, lb, ub = state["arrays"]
        x, objective = state["x"], state["objective"]
        opf.global_update_static(case["n"], off.data_ptr(), u.data_ptr(), c.data_ptr(), lb.data_ptr(), ub.data_ptr(),
                                 RHO, x.data_ptr(), objective.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"x": x, "objective": objective}
    if kind == "serve":
        server, requests = state["server"], state["requests"]
        for tag, (model, lp, lq) in enumerate(requests):
            server.submit(model, lp, lq, tag)
        objective = np.zeros(len(requests))
        waiting = len(requests)
        while waiting:
            server.step()
            for done in server.poll():
                objective[done["tag"]] = done["objective"]
                waiting -= 1
        x = [server.take_solution(tag, model) for tag, (model, _, _) in enumerate(requests)]
        return _handed_on(case, np.concatenate(x), objective)
    how = dict(rho=RHO, eps_rel=case["eps_rel"], eps_abs_pres=case.get("eps_abs", EPS_ABS),
               max_iter=case["max_iter"], check_every=case["check_every"], precision=PRECISION[case["precision"]])
    if kind == "batch":
        batch = state["batch"]
        batch.set_loads(0, state["lp"].numpy(), state["lq"].numpy())
        batch.solve(**how)
        x, objective = batch.solution(out=(state["x"].numpy(), state["objective"].numpy()))
        return _handed_on(case, x, objective)
    solver = state["solver"]
    if kind == "solve":
        solver.set_loads(state["lp"], state["lq"])
    solver.precompute()
    solver.solve(**how)
    return _handed_on(case, *solver.solution())


# ------------------------------------------------- plain 64-bit counterpart
def _phases(mask):
    return [p for p in range(3) if (int(mask) >> p) & 1]


def _feeder_lp(f):
    """Linearized three-phase power flow of a feeder with constant-power wye loads, no shunts and unit taps:
    costs, bounds, voltage marks and the blocks (variables, rows, load behind each right-hand side)."""
    c, lb, ub, volt, var = [], [], [], [], {}

    def add(key, lo, hi, cost=0.0, is_volt=False):
        var[key] = len(c)
        c.append(cost)
        lb.append(lo)
        ub.append(hi)
        volt.append(is_volt)

    nb = int(f["n_bus"])
    for g, mask in enumerate(f["gen_phases"]):
        for p in _phases(mask):
            add(("gp", g, p), f["gen_pmin"][g, p], f["gen_pmax"][g, p], f["gen_cost"][g])
            add(("gq", g, p), f["gen_qmin"][g, p], f["gen_qmax"][g, p])
    for i in range(nb):
        for p in _phases(f["bus_phases"][i]):
            add(("w", i, p), f["bus_wmin"][i, p], f["bus_wmax"][i, p], 0.0, True)
    for l, mask in enumerate(f["load_phases"]):
        for p in _phases(mask):
            for field in ("pb", "qb", "pd", "qd"):
                add((field, l, p), -math.inf, math.inf)
    for e, mask in enumerate(f["line_phases"]):
        for p in _phases(mask):
            for field in ("pij", "qij", "pji", "qji"):
                add((field, e, p), -math.inf, math.inf)
    out, into, loads, gens = ([[] for _ in range(nb)] for _ in range(4))
    for e in range(len(f["line_from"])):
        out[f["line_from"][e]].append(e)
        into[f["line_to"][e]].append(e)
    for l, i in enumerate(f["load_bus"]):
        loads[i].append(l)
    for g, i in enumerate(f["gen_bus"]):
        gens[i].append(g)
    on_line = [_phases(m) for m in f["line_phases"]]
    on_load = [_phases(m) for m in f["load_phases"]]
    on_gen = [_phases(m) for m in f["gen_phases"]]

    def bus_rows(i):
        rows, names = [], [("w", i, p) for p in _phases(f["bus_phases"][i])]
        for p in _phases(f["bus_phases"][i]):
            for s in "pq":
                row = {(s + "ij", e, p): 1.0 for e in out[i] if p in on_line[e]}
                row.update({(s + "ji", e, p): 1.0 for e in into[i] if p in on_line[e]})
                row.update({(s + "b", l, p): 1.0 for l in loads[i] if p in on_load[l]})
                row.update({("g" + s, g, p): -1.0 for g in gens[i] if p in on_gen[g]})
                rows.append((row, -1))
        for l in loads[i]:
            for p in on_load[l]:
                for k, s in enumerate("pq"):
                    rows.append(({(s + "d", l, p): 1.0}, 2 * (3 * l + p) + k))
                    rows.append(({(s + "b", l, p): 1.0, (s + "d", l, p): -1.0}, -1))
        return rows, names

    def line_rows(e):
        rows, i, j = [], f["line_from"][e], f["line_to"][e]
        r, x = f["line_r"][e], f["line_x"][e]
        for p in on_line[e]:
            for s in "pq":
                rows.append(({(s + "ij", e, p): 1.0, (s + "ji", e, p): 1.0}, -1))
            row = {("w", i, p): 1.0, ("w", j, p): -1.0}
            for q in on_line[e]:
                turn = 0.0 if q == p else (-1.0 if (q - p) % 3 == 1 else 1.0) * math.sqrt(3.0)
                lead = -2.0 if q == p else 1.0
                row["pij", e, q] = lead * r[p, q] + turn * x[p, q]
                row["qij", e, q] = lead * x[p, q] - turn * r[p, q]
            rows.append((row, -1))
        return rows

    blocks = []

    def block(rows, names):
        idx = sorted({var[k] for row, _ in rows for k in row} | {var[k] for k in names})
        at = {v: n for n, v in enumerate(idx)}
        a = np.zeros((len(rows), len(idx)))
        for n, (row, _) in enumerate(rows):
            for key, value in row.items():
                a[n, at[var[key]]] += value
        blocks.append((np.array(idx), a, np.array([source for _, source in rows])))

    leaf = [i > 0 and not out[i] for i in range(nb)]
    for i in range(nb):
        if not leaf[i]:
            block(*bus_rows(i))
    for e in range(len(on_line)):
        rows, names = line_rows(e), []
        if leaf[f["line_to"][e]]:
            more, names = bus_rows(f["line_to"][e])
            rows = rows + more
        block(rows, names)
    return np.array(c), np.array(lb), np.array(ub), np.array(volt), blocks


class _Lp:
    """Costs, bounds, start point and, stacked over the blocks, M = I - A^+ A (entries) and each A^+."""

    def __init__(self, c, lb, ub, volt, blocks):
        self.c, self.lb, self.ub, self.blocks = c, lb, ub, blocks
        mid = np.where(np.isfinite(lb), lb, np.where(np.isfinite(ub), ub, 0.0))
        both = np.isfinite(lb) & np.isfinite(ub)
        mid[both] = 0.5 * (lb[both] + ub[both])
        self.x0 = np.where(volt, 1.0, mid)
        self.idx = np.concatenate([i for i, _, _ in blocks])
        self.pinv, rows, cols, vals, at = [], [], [], [], 0
        self.sum_nf = 0
        for i, a, _ in blocks:
            n = len(i)
            p = np.linalg.pinv(a, rcond=1e-11) if a.size else np.zeros((n, 0))
            m = np.eye(n) - p @ a
            null = int(round(np.trace(m)))
            self.sum_nf += n * min(null, n - null)
            self.pinv.append(p)
            r, k = np.meshgrid(np.arange(at, at + n), np.arange(at, at + n), indexing="ij")
            rows.append(r.ravel())
            cols.append(k.ravel())
            vals.append(m.ravel())
            at += n
        self.slots = at
        self.rows, self.cols, self.vals = (np.concatenate(v) for v in (rows, cols, vals))
        self.a_values = sum(a.size for _, a, _ in blocks)

    def bbar(self, rhs):
        """A^+ b of every block; rhs(sources) gives a block's right-hand sides, one column per instance."""
        return np.concatenate([p @ rhs(s) for p, (_, _, s) in zip(self.pinv, self.blocks)])


@functools.lru_cache(maxsize=4)
def _feeder_model(buses, seed):
    return _Lp(*_feeder_lp(_feeder(buses, seed)))


def _load_rhs(lp, lq):
    """Right-hand sides of rows from scenario loads [count, n_load, 3]: source 2 * (3 * load + phase) + (0: p, 1: q)."""
    both = np.stack([lp.reshape(len(lp), -1), lq.reshape(len(lq), -1)], axis=2).reshape(len(lp), -1).T

    def rhs(sources):
        return np.where(sources[:, None] >= 0, both[np.maximum(sources, 0)], 0.0)

    return rhs


def _admm(m, bbar, case, again):
    """Algorithm 1 in 64 bits, one column per instance, each to its own stop: the test of Sec. III-C every
    check_every iterations (or the budget) and, with again > 0, on from there until it holds again, tested every
    `again` iterations for the length of the polish.  Returns x, a row per instance."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    count, g = bbar.shape[1], len(m.c)

    def t(v):
        return torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)

    order = np.argsort(m.rows, kind="stable")
    starts = np.concatenate([[0], np.cumsum(np.bincount(m.rows, minlength=m.slots))])
    mat = torch.sparse_csr_tensor(torch.as_tensor(starts, device=dev), torch.as_tensor(m.cols[order], device=dev),
                                  t(m.vals[order]), (m.slots, m.slots))
    idx = torch.as_tensor(m.idx, device=dev)
    by_global = np.argsort(m.idx, kind="stable")
    copies = np.bincount(m.idx, minlength=g)
    gather = torch.sparse_csr_tensor(torch.as_tensor(np.concatenate([[0], np.cumsum(copies)]), device=dev),
                                     torch.as_tensor(by_global, device=dev),
                                     torch.ones(m.slots, dtype=torch.float64, device=dev), (g, m.slots))
    c, lb, ub, per, bbar = t(m.c)[:, None], t(m.lb)[:, None], t(m.ub)[:, None], 1.0 / (RHO * t(copies)[:, None]), t(bbar)
    xs = t(m.x0)[idx][:, None].repeat(1, count)
    lam = torch.zeros_like(xs)
    result = torch.zeros((g, count), dtype=torch.float64, device=dev)
    k, cap = case["check_every"], (case["max_iter"] + case["check_every"] - 1) // case["check_every"] * case["check_every"]
    first = np.full(count, -1)        # iteration at which the first test held
    done = np.zeros(count, dtype=bool)
    it = 0
    while not done.all():
        it += 1
        x = torch.clamp((gather @ (RHO * xs - lam) - c) * per, lb, ub)
        bx = x[idx]
        v = bx + lam / RHO
        new = mat @ v + bbar
        lam = lam + RHO * (bx - new)
        old, xs = xs, new
        main, polish = it % k == 0 and (first < 0).any(), again > 0 and (first >= 0).any()
        if not (main or polish):
            continue
        norm = [torch.linalg.vector_norm(w, dim=0).cpu().numpy() for w in (bx - new, new - old, bx, new, lam)]
        held = ((norm[0] <= case["eps_rel"] * np.maximum(norm[2], norm[3])) & (RHO * norm[1] <= case["eps_rel"] * norm[4])
                & (norm[0] <= case.get("eps_abs", EPS_ABS)))
        stop = np.zeros(count, dtype=bool)
        if polish:
            since = it - first
            length = 2 * k if again < k else k
            stop |= ~done & (first >= 0) & (since % again == 0) & (held | ((since >= length) & (it >= cap)))
        if main:
            now = (first < 0) & (held | (it >= cap))
            first[now] = it
            if again == 0:
                stop |= now
        if stop.any():
            at = torch.as_tensor(np.nonzero(stop)[0], device=dev)
            result[:, at] = x[:, at]
            done |= stop
    return result.T.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "update":
        off, u, c, lb, ub = _update_arrays(case, seed)
        copies = (off[1:] - off[:-1]).long()
        owner = torch.repeat_interleave(torch.arange(case["n"], device=u.device), copies)
        total = torch.zeros(case["n"], dtype=torch.float64, device=u.device).index_add_(0, owner, u)
        x = torch.minimum(torch.maximum((total - c) / (RHO * copies), lb), ub)
        return {"x": x, "objective": (c * x).sum().reshape(1)}
    if kind == "consensus":
        g = _consensus(case, seed)
        m = _Lp(g["c"], g["lb"], g["ub"], np.zeros(len(g["c"]), dtype=bool),
                [(s["idx"], s["A"], s["b"]) for s in g["subs"]])
        again = case["check_every"] if case["precision"] == "mixed" else 0
        x = _admm(m, m.bbar(lambda b: b[:, None]), case, again)[0]
        return {"x": x, "objective": float(x @ torch.as_tensor(m.c, device=x.device))}
    if kind == "serve":
        xs, objective = [], []
        for key, buses, feeder_seed in SERVED:
            if case[key]:
                m = _feeder_model(buses, feeder_seed)
                rhs = _load_rhs(*_scenarios(_feeder(buses, feeder_seed), seed + buses, case[key]))
                x = _admm(m, m.bbar(rhs), case, 2 if case["eps_rel"] > 0 else 0)
                xs.append(x.reshape(-1))
                objective.append(x @ torch.as_tensor(m.c, device=x.device))
        return {"x": torch.cat(xs), "objective": torch.cat(objective)}
    m = _feeder_model(case["buses"], case["seed"])
    count = case.get("instances", 1)
    rhs = _load_rhs(*_scenarios(_feeder(case["buses"], case["seed"]), seed, count))
    again = 0 if case["precision"] == "fp64" else 2 if kind == "batch" else case["check_every"]
    x = _admm(m, m.bbar(rhs), case, again)
    objective = x @ torch.as_tensor(m.c, device=x.device)
    return {"x": x[0], "objective": float(objective[0])} if kind == "solve" else {"x": x, "objective": objective}


# --------------------------------------------------------------------- work
def work(case):
    """Per iteration and instance: two products with each block's projector factor (the smaller of row space and
    null space), the slots' updates and the globals'; the data of the problem and its solution once."""
    kind = case["kind"]
    if kind == "update":
        return {"bytes": case["n"] * (4 + 8 * 2 + 8 * 4), "flops": case["n"] * 7}
    if kind == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        nominal = {"r13": 4200, "r34": 12500, "r123": 38000}
        for key, buses, feeder_seed in SERVED:
            one = dict(case, kind="batch", buses=buses, seed=feeder_seed, instances=case[key],
                       iters=nominal[key] if case["eps_rel"] > 0 else case["max_iter"])
            if case[key]:
                total = {k: total[k] + v for k, v in work(one).items()}
        return total
    if kind == "consensus":
        # blocks of 2 .. widest slots with 1 .. n_s - 1 rows: on average n_s min(m_s, n_s - m_s) is n_s^2 / 4
        w = case["widest"]
        slots = case["blocks"] * (w + 2) / 2
        sum_nf = case["blocks"] * sum(n * n for n in range(2, w + 1)) / (4 * (w - 1))
        globals_, data = case["n"], 2 * sum_nf
    else:
        m = _feeder_model(case["buses"], case["seed"])
        slots, sum_nf, globals_, data = m.slots, m.sum_nf, len(m.c), m.a_values
    count = case.get("instances", 1)
    loads = 0 if kind == "consensus" else 6 * len(_feeder(case["buses"], case["seed"])["load_bus"])
    return {"bytes": 8.0 * (data + 3 * globals_ + count * (loads + globals_ + 1)),
            "flops": float(count) * case["iters"] * (4.0 * sum_nf + 8.0 * slots + 2.0 * globals_)}
