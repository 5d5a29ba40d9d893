"""What this framework is used for, as cases that can be timed and compared.

A case is one call pattern of a user's program on one 0-1 ILP (or several):
running the dual iterations on a resident instance and reading the bound and
the multipliers, solving to a rounded point, solving a batch, serving a stream
of requests, solving from host arrays, reading the dual state, and reducing
caller-held energies.  The ILPs have the shapes of the paper's workloads: MAP
inference on grid MRFs, graph matching with product terms, cell tracking, and
packing rows with small integer coefficients.  All are synthetic and seeded.

`listed()` holds the fixed cases, `draw()` gives more of the same ranges,
`prepare()` makes inputs and plan, `run()` is one pass through the public entry
points, `work()` states what a pass cannot do without, and `exact()` computes
the same results in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_2111_10270_gb300 as fdog

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a parity-sized grid, a handful of iterations, multipliers read back
        {"name": "grid_8x8x3_iterate", "op": "iterate", "family": "grid", "h": 8, "w": 8, "labels": 3, "iters": 20},
        # an image-sized grid with a ragged label count, run to the usual cap of 500 iterations
        {"name": "grid_100x150x5_iterate", "op": "iterate", "family": "grid", "h": 100, "w": 150, "labels": 5,
         "iters": 500},
        # a whole solve of the large grid: dual iterations, rounding, objective, solution
        {"name": "grid_512x512x4_solve", "op": "solve", "family": "grid", "h": 512, "w": 512, "labels": 4,
         "iters": 500},
        # graph matching whose product terms join neighbouring matches only
        {"name": "matching_500_iterate", "op": "iterate", "family": "matching", "left": 500, "dense": False,
         "iters": 200},
        # the same matching with every candidate pair of neighbouring nodes: rows over hundreds of copies
        {"name": "matching_500_dense_bound", "op": "bound", "family": "matching", "left": 500, "dense": True,
         "iters": 100},
        # one cell-tracking sequence: flow rows of many lengths
        {"name": "cells_20x600_iterate", "op": "iterate", "family": "cells", "frames": 20, "dets": 600, "iters": 200},
        # several sequences solved together
        {"name": "cells_batch_12", "op": "batch", "family": "cells", "count": 12, "frames": 30, "dets": 900,
         "iters": 500},
        # a mixed request stream through the continuous-batching server, each request from its host arrays
        {"name": "serve_16", "op": "serve", "family": "mixed", "count": 16, "iters": 500},
        # one request from host arrays to a rounded point: create, plan, upload, solve, read back
        {"name": "grid_128x128x4_from_host", "op": "from_host", "family": "grid", "h": 128, "w": 128, "labels": 4,
         "iters": 500},
        # reading a resident dual state: both bounds and every min-marginal
        {"name": "grid_256x256x4_read", "op": "read", "family": "grid", "h": 256, "w": 256, "labels": 4, "iters": 50},
        # packing rows with small integer coefficients: wide BDDs on the general kernels, default stream
        {"name": "packing_40k_iterate", "op": "iterate", "family": "packing", "vars": 30011, "rows": 40007,
         "iters": 50},
        # a caller's own energies reduced without allocating
        {"name": "reduce_4M", "op": "reduce", "family": "values", "n": 4000037},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.randrange(12)
    if kind == 0:
        return {"op": "iterate", "family": "grid", "h": _log_int(rng, 4, 30), "w": _log_int(rng, 4, 30),
                "labels": rng.randint(2, 6), "iters": rng.randint(20, 60)}
    if kind == 1:
        h, w = _log_int(rng, 40, 220), _log_int(rng, 40, 220)
        labels = rng.randint(2, min(8, max(2, int(math.sqrt(400000 / (h * w))))))
        return {"op": "iterate", "family": "grid", "h": h, "w": w, "labels": labels, "iters": rng.randint(100, 500)}
    if kind == 2:
        h, w = _log_int(rng, 150, 512), _log_int(rng, 150, 512)
        return {"op": "solve", "family": "grid", "h": h, "w": w, "labels": rng.randint(2, 4),
                "iters": rng.randint(200, 500)}
    if kind == 3:
        return {"op": "iterate", "family": "matching", "left": _log_int(rng, 50, 1000), "dense": False,
                "iters": rng.randint(100, 200)}
    if kind == 4:
        return {"op": "bound", "family": "matching", "left": _log_int(rng, 80, 500), "dense": True,
                "iters": rng.randint(50, 100)}
    if kind == 5:
        return {"op": "iterate", "family": "cells", "frames": rng.randint(5, 40), "dets": _log_int(rng, 80, 1200),
                "iters": rng.randint(100, 200)}
    if kind == 6:
        return {"op": "batch", "family": "cells", "count": rng.randint(3, 12), "frames": rng.randint(6, 30),
                "dets": _log_int(rng, 100, 900), "iters": rng.randint(200, 500)}
    if kind == 7:
        return {"op": "serve", "family": "mixed", "count": rng.randint(5, 16), "iters": rng.randint(200, 500)}
    if kind == 8:
        return {"op": "from_host", "family": "grid", "h": _log_int(rng, 20, 200), "w": _log_int(rng, 20, 200),
                "labels": rng.randint(2, 4), "iters": rng.randint(200, 500)}
    if kind == 9:
        return {"op": "read", "family": "grid", "h": _log_int(rng, 30, 256), "w": _log_int(rng, 30, 256),
                "labels": rng.randint(2, 4), "iters": rng.randint(20, 50)}
    if kind == 10:
        rows = _log_int(rng, 2000, 40000)
        return {"op": "iterate", "family": "packing", "vars": max(400, int(rows * rng.uniform(0.5, 1.0))),
                "rows": rows, "iters": rng.randint(20, 50)}
    return {"op": "reduce", "family": "values", "n": _log_int(rng, 2000, 8000000)}


# ---------------------------------------------------------------------------
# the ILPs: host arrays in the form the library's create call takes.  Points, candidates and supports follow from
# the sizes, so that a case has the same rows under every seed; the costs come from the seed.
# ---------------------------------------------------------------------------
def _ilp(cost, lens, col, coef, sense, rhs):
    row_ptr = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    return {"n_vars": len(cost), "cost": np.asarray(cost, np.float64), "row_ptr": row_ptr,
            "col": np.asarray(col, np.int32), "coef": np.asarray(coef, np.int32), "sense": np.asarray(sense, np.int8),
            "rhs": np.asarray(rhs, np.int64)}


def _grid(h, w, labels, seed):
    """MAP inference on an h x w four-connected grid: a simplex row per node, 2 * labels marginalisation rows
    per edge; unary costs N(0, 1), Potts weights U(0, 2)."""
    rng = np.random.default_rng(seed)
    L, U = labels, h * w
    node = torch.arange(U, device=DEV).reshape(h, w)
    right = torch.stack([node[:, :-1], node[:, 1:]], -1).reshape(-1, 2)
    down = torch.stack([node[:-1], node[1:]], -1).reshape(-1, 2)
    E = torch.cat([right, down])
    E = E[torch.argsort(E[:, 0], stable=True)]
    nE = len(E)
    lab = torch.arange(L, device=DEV)
    y = U * L + torch.arange(nE * L * L, device=DEV).reshape(nE, L, L)
    side0 = torch.cat([(E[:, :1] * L + lab)[:, :, None], y], 2)                  # [edge, label, x and its y]
    side1 = torch.cat([(E[:, 1:] * L + lab)[:, :, None], y.transpose(1, 2)], 2)
    marg = torch.stack([side0, side1], 1).reshape(-1)
    col = torch.cat([torch.arange(U * L, device=DEV), marg]).to(torch.int32).cpu().numpy()
    coef = np.ones(len(col), np.int32)
    coef[U * L::L + 1] = -1
    potts = (1.0 - np.eye(L)).reshape(-1)
    cost = np.concatenate([rng.standard_normal(U * L),
                           (rng.uniform(0.0, 2.0, nE)[:, None] * potts[None]).reshape(-1)])
    lens = np.concatenate([np.full(U, L), np.full(nE * 2 * L, L + 1)])
    rhs = np.concatenate([np.ones(U, np.int64), np.zeros(nE * 2 * L, np.int64)])
    return _ilp(cost, lens, col, coef, np.zeros(len(lens), np.int8), rhs)


def _nearest(a, b, k):
    a, b = torch.from_numpy(a).to(DEV), torch.from_numpy(b).to(DEV)
    return torch.cdist(a, b).topk(min(k, len(b)), largest=False).indices.cpu().numpy()


def _matching(left, dense, seed):
    """Graph matching, twice as many right nodes, 20 candidates each: at most one match per node, and for
    neighbouring left nodes a product variable per candidate pair (all pairs, or neighbouring ones)."""
    rng = np.random.default_rng([left, dense])
    right, cand_n, knn = 2 * left, min(20, 2 * left), 10
    P, R = rng.random((left, 2)), rng.random((right, 2))
    cand = np.argsort(rng.random((left, right)), axis=1)[:, :cand_n]
    near = _nearest(P, P, knn + 1)[:, 1:]
    p, q = np.repeat(np.arange(left), near.shape[1]), near.reshape(-1)
    pairs = np.unique(np.stack([np.minimum(p, q), np.maximum(p, q)], 1)[p != q], axis=0)
    A, B = cand[pairs[:, 0]][:, :, None], cand[pairs[:, 1]][:, None, :]
    ok = A != B
    if not dense:
        rn = _nearest(R, R, knn + 1)[:, 1:]
        close = np.zeros((right, right), bool)
        close[np.repeat(np.arange(right), rn.shape[1]), rn.reshape(-1)] = True
        ok &= close[A, B]
    pi, ia, ib = np.nonzero(ok)
    x = np.arange(left * cand_n).reshape(left, cand_n)
    xa, xb = x[pairs[pi, 0], ia], x[pairs[pi, 1], ib]
    z = x.size + np.arange(len(xa))
    node = cand.reshape(-1)
    order = np.argsort(node, kind="stable")
    degree = np.bincount(node, minlength=right)
    kept = degree >= 2
    right_cols = order[kept[node[order]]]
    products = np.stack([xa, z, xb, z, xa, xb, z], 1).reshape(-1)
    col = np.concatenate([x.reshape(-1), right_cols, products])
    coef = np.concatenate([np.ones(x.size + len(right_cols)), np.tile([-1, 1, -1, 1, 1, 1, -1], len(z))])
    lens = np.concatenate([np.full(left, cand_n), degree[kept], np.tile([2, 2, 3], len(z))])
    rhs = np.concatenate([np.ones(left + kept.sum()), np.tile([0, 0, 1], len(z))])
    cost = np.random.default_rng(seed).standard_normal(x.size + len(z))
    return _ilp(cost, lens, col, coef, np.full(len(lens), -1), rhs)


def _cells(frames, dets, seed):
    """Cell tracking: detections, transitions to the 5 nearest detections of the next frame, one division into
    the 2 nearest; out-flow and in-flow rows, and at most one detection of close triples."""
    rng = np.random.default_rng([frames, dets])
    count = np.maximum(8, (dets * rng.uniform(0.5, 1.5, frames)).astype(np.int64))
    off = np.concatenate([[0], np.cumsum(count)])
    pts = [rng.random((c, 2)) for c in count]
    n_det, src = int(off[-1]), np.arange(int(off[-2]))
    near = np.concatenate([_nearest(pts[f], pts[f + 1], 5) + off[f + 1] for f in range(frames - 1)])
    t_var = n_det + np.arange(5 * len(src)).reshape(-1, 5)
    d_var = n_det + t_var.size + np.arange(len(src))
    out = np.concatenate([src[:, None], t_var, d_var[:, None]], 1)
    dst = np.concatenate([near.reshape(-1), near[:, :2].reshape(-1)])
    into = np.concatenate([t_var.reshape(-1), np.repeat(d_var, 2)])
    order = np.lexsort((into, dst))
    degree = np.bincount(dst, minlength=n_det)
    has = np.flatnonzero(degree)
    lens_in = degree[has] + 1
    at = np.concatenate([[0], np.cumsum(lens_in)])[:-1]
    col_in, coef_in = np.empty(lens_in.sum(), np.int64), np.ones(lens_in.sum(), np.int64)
    head = np.zeros(len(col_in), bool)
    head[at] = True
    col_in[head], col_in[~head], coef_in[head] = has, into[order], -1
    triples = []
    for f in range(frames):
        used = np.zeros(count[f], bool)
        for a, b, c in _nearest(pts[f], pts[f], 3).tolist():
            if len({a, b, c}) == 3 and not (used[a] or used[b] or used[c]):
                used[[a, b, c]] = True
                triples.append(sorted((a + off[f], b + off[f], c + off[f])))
    triples = np.asarray(triples, np.int64).reshape(-1, 3)
    col = np.concatenate([out.reshape(-1), col_in, triples.reshape(-1)])
    coef = np.concatenate([np.tile([-1] + [1] * 6, len(src)), coef_in, np.ones(triples.size)])
    lens = np.concatenate([np.full(len(src), 7), lens_in, np.full(len(triples), 3)])
    rhs = np.concatenate([np.zeros(len(src) + len(lens_in)), np.ones(len(triples))])
    cost = np.random.default_rng(seed).standard_normal(n_det + t_var.size + len(d_var))
    return _ilp(cost, lens, col, coef, np.full(len(lens), -1), rhs)


def _packing(n_vars, n_rows, seed):
    """Packing rows of 4 to 12 variables: coefficients 1 to 3 after one of 24 patterns, capacity near half the
    row's sum (no row forces a variable or accepts every assignment)."""
    rng = np.random.default_rng([n_vars, n_rows])
    pats = [rng.integers(1, 4, int(k)) for k in rng.integers(4, 13, 24)]
    kind = rng.integers(0, len(pats), n_rows)
    lens = np.array([len(p) for p in pats])[kind]
    ptr = np.concatenate([[0], np.cumsum(lens)])
    col, coef = np.empty(ptr[-1], np.int64), np.empty(ptr[-1], np.int64)
    rhs = np.empty(n_rows, np.int64)
    for k, p in enumerate(pats):
        rows = np.flatnonzero(kind == k)
        # distinct ascending variables: a start and strictly positive gaps, wrapped into the range
        gaps = rng.integers(1, max(2, n_vars // 16), (len(rows), len(p)))
        gaps[:, 0] = 0
        v = np.sort((rng.integers(0, n_vars, len(rows))[:, None] + np.cumsum(gaps, 1)) % n_vars, axis=1)
        slots = ptr[rows][:, None] + np.arange(len(p))
        col[slots], coef[slots] = v, p
        rhs[rows] = max(int(p.max()), int(p.sum()) // 2)
    return _ilp(-np.random.default_rng(seed).exponential(1.0, n_vars), lens, col, coef, np.full(n_rows, -1), rhs)


def _mixed(count, i, seed):
    """Request i of a stream: grids of side 16 to 160 and 2 to 6 labels, matchings of 50 to 800 left nodes."""
    at = (0.5 + i * 0.618033988749895) % 1.0
    if i % 2 == 0:
        side = int(16 * 10.0 ** at)
        return _grid(side, side, 2 + (i // 2) % 5, seed)
    return _matching(int(50 * 16.0 ** at), False, seed)


def _inputs(case, seed):
    if case["family"] == "grid":
        return [_grid(case["h"], case["w"], case["labels"], seed)]
    if case["family"] == "matching":
        return [_matching(case["left"], case["dense"], seed)]
    if case["family"] == "packing":
        return [_packing(case["vars"], case["rows"], seed)]
    n = case.get("count", 1)
    if case["family"] == "cells":
        # the sequences of a batch are 0.4 to 1.6 times as long as its nominal length
        frames = [max(4, int(case["frames"] * (0.4 + 1.2 * (i + 0.5) / n))) for i in range(n)]
        return [_cells(f, case["dets"], seed * 1009 + i) for i, f in enumerate(frames)]
    return [_mixed(n, i, seed * 1009 + i) for i in range(n)]


def _create(g, **params):
    return fdog.Instance(g["n_vars"], g["cost"], g["row_ptr"], g["col"], g["coef"], g["sense"], g["rhs"], **params)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _row_order(inst, g):
    """Where each of the instance's slots stands in the caller's rows (None: they come in that order)."""
    var, row, _ = inst.multipliers()
    key = row.astype(np.int64) * g["n_vars"] + var
    return None if bool(np.all(key[1:] > key[:-1])) else np.argsort(key, kind="stable")


def prepare(case, seed):
    op = case["op"]
    if op == "reduce":
        gen = torch.Generator(DEV).manual_seed(seed)
        v = torch.randn(case["n"], generator=gen, device=DEV, dtype=torch.float64)
        return {"op": op, "values": v, "out": torch.zeros(1, device=DEV, dtype=torch.float64)}
    ilps = _inputs(case, seed)
    s = {"op": op, "iters": case["iters"]}
    if op == "serve":
        return dict(s, ilps=ilps, server=fdog.Server(max_iters=case["iters"]))
    # packing runs on the default stream, the others on a stream of their own
    s["stream"] = None if case["family"] == "packing" else torch.cuda.Stream()
    if op == "from_host":
        return dict(s, ilps=ilps)
    fixed = op in ("iterate", "bound", "read")  # a fixed number of iterations; else the stopping rule of 1e-4
    s["insts"] = [_create(g, tol=0.0 if fixed else 1e-4).build(0, s["stream"]) for g in ilps]
    if op == "iterate":
        s["order"] = _row_order(s["insts"][0], ilps[0])
    elif op == "read":
        s["insts"][0].iterate(case["iters"])
    elif op == "batch":
        s["batch"] = fdog.Batch(s["insts"], s["stream"])
    return s


def _solve(inst, iters):
    done, lb = inst.iterate(iters)
    status, rounds = inst.primal_round()
    x, objective, feasible = inst.solution()
    return {"iters": done, "lb": lb, "status": status, "rounds": rounds, "x": x, "objective": objective,
            "feasible": feasible}


def run(state):
    op = state["op"]
    if op == "reduce":
        v = state["values"]
        rc = fdog.lib().fdog_bound_reduce_noalloc(v.data_ptr(), v.numel(), 1.25, state["out"].data_ptr(),
                                                  torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise RuntimeError("fdog_bound_reduce_noalloc: %d" % rc)
        return {"sum": state["out"]}
    if op == "serve":
        server = state["server"]
        tickets = [server.submit(_create(g, tol=1e-4)) for g in state["ilps"]]
        got = []
        for t in tickets:
            if not server.wait(t):
                raise RuntimeError("request %d timed out" % t)
            status = server.poll(t)["status"]
            inst = server.take(t)
            x, objective, feasible = inst.solution()
            inst.close()
            got.append((status, x, objective, feasible))
        return {"status": np.array([g[0] for g in got]), "x": np.concatenate([g[1] for g in got]),
                "objective": np.array([g[2] for g in got]), "feasible": np.array([g[3] for g in got])}
    if op == "from_host":
        inst = _create(state["ilps"][0], tol=1e-4).build(0, state["stream"])
        got = _solve(inst, state["iters"])
        inst.close()
        return got
    if op == "batch":
        for inst in state["insts"]:
            inst.reset()
        iters, rounds, status = state["batch"].solve(state["iters"])
        got = [inst.solution() for inst in state["insts"]]
        return {"iters": iters, "rounds": rounds, "status": status, "x": np.concatenate([g[0] for g in got]),
                "objective": np.array([g[1] for g in got]), "feasible": np.array([g[2] for g in got])}
    inst = state["insts"][0]
    if op == "read":
        running, feasible = inst.lower_bound()
        var, row, m0, m1 = inst.min_marginals()
        return {"lb": running, "lb_feasible": feasible, "var": var, "row": row, "m0": m0, "m1": m1}
    inst.reset()
    if op == "solve":
        return _solve(inst, state["iters"])
    done, lb = inst.iterate(state["iters"])
    if op == "bound":
        running, feasible = inst.lower_bound()
        return {"iters": done, "lb": lb, "lb_running": running, "lb_feasible": feasible}
    _, _, lam = inst.multipliers()
    return {"iters": done, "lb": lb, "lam": lam if state["order"] is None else lam[state["order"]]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _sizes(family, case, i=0):
    """(variables, slots) of a case's ILP, to within a few per cent."""
    if family == "grid":
        h, w, L = case["h"], case["w"], case["labels"]
        e = h * (w - 1) + w * (h - 1)
        return h * w * L + e * L * L, h * w * L + e * 2 * L * (L + 1)
    if family == "matching":
        x = case["left"] * min(20, 2 * case["left"])
        z = 5.8 * case["left"] * 400 * (1.0 if case["dense"] else 10.0 / (2 * case["left"]))
        return x + z, 2 * x + 7 * z
    if family == "cells":
        d = case["frames"] * case["dets"] * case.get("count", 1)
        return 7 * d, 16 * d
    if family == "packing":
        return case["vars"], 8 * case["rows"]
    at = (0.5 + i * 0.618033988749895) % 1.0
    if i % 2 == 0:
        side = int(16 * 10.0 ** at)
        return _sizes("grid", {"h": side, "w": side, "labels": 2 + (i // 2) % 5})
    return _sizes("matching", {"left": int(50 * 16.0 ** at), "dense": False})


def work(case):
    """Per pass of Alg. 1 (two per iteration): every slot's multiplier read and written and its variable's index
    read, and the term of every variable read once; about ten additions and minima per slot.  A read of the state
    and a solution add their own bytes once."""
    if case["op"] == "reduce":
        return {"bytes": 8 * case["n"] + 8, "flops": case["n"]}
    n, s = 0, 0
    for i in range(case["count"] if case["family"] == "mixed" else 1):
        a, b = _sizes(case["family"], case, i)
        n, s = n + a, s + b
    if case["op"] == "read":
        # multipliers and terms in for the bounds and the min-marginals, four arrays of slots out
        return {"bytes": (4 + 4 + 16) * s + 4 * n, "flops": 20 * s}
    end = {"iterate": 12 * s, "bound": 4 * s + 4 * n}.get(case["op"], n)
    return {"bytes": 2 * case["iters"] * (12 * s + 4 * n) + end, "flops": 2 * case["iters"] * 10 * s}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
class _Rows64:
    """Rows of one pattern (coefficients, sense, right-hand side): shortest paths over their partial sums."""

    def __init__(self, coef, sense, rhs, slots, var):
        self.slots, self.var, self.k = slots, var, len(coef)  # slots, var: [layer, row]
        ends = {0}
        reach = [ends]
        for a in coef:
            ends = ends | {s + a for s in ends}
            reach.append(ends)
        good = {s for s in reach[-1] if (sense > 0 or s <= rhs) and (sense < 0 or s >= rhs)}
        layers = [sorted(good)]
        for t in range(self.k - 1, -1, -1):
            good = {s for s in reach[t] if s in good or s + coef[t] in good}
            layers.append(sorted(good))
        layers.reverse()

        def at(frm, shift, to):
            pos = {s: i for i, s in enumerate(to)}
            return torch.tensor([pos.get(s + shift, len(to)) for s in frm], device=DEV)

        self.lo = [at(layers[t], 0, layers[t + 1]) for t in range(self.k)]
        self.hi = [at(layers[t], coef[t], layers[t + 1]) for t in range(self.k)]
        self.from_lo = [at(layers[t + 1], 0, layers[t]) for t in range(self.k)]
        self.from_hi = [at(layers[t + 1], -coef[t], layers[t]) for t in range(self.k)]
        m = slots.shape[1]
        self.inf = torch.full((1, m), math.inf, dtype=torch.float64, device=DEV)
        self.root = torch.cat([torch.zeros((1, m), dtype=torch.float64, device=DEV), self.inf])
        self.top = torch.cat([torch.zeros((len(layers[-1]), m), dtype=torch.float64, device=DEV), self.inf])

    def _step(self, x, a, b, lam):
        return torch.cat([torch.minimum(x[a], x[b] + lam), self.inf])

    def down(self, B, t, lam):
        return self._step(B, self.lo[t], self.hi[t], lam)

    def up(self, F, t, lam):
        return self._step(F, self.from_lo[t], self.from_hi[t], lam)

    def marginals(self, F, B, t, lam):
        F = F[:-1]
        return (F + B[self.lo[t]]).amin(0), (F + B[self.hi[t]]).amin(0) + lam

    def labels(self, lam, forward):
        x = [self.root if forward else self.top]
        for t in range(self.k) if forward else range(self.k - 1, -1, -1):
            x.append(self.up(x[-1], t, lam[t]) if forward else self.down(x[-1], t, lam[t]))
        return x if forward else x[::-1]

    def sweep(self, lam, T, omega, forward):
        """One pass; lam [layer, row] is updated, the rows' shares of the lifted bound come back."""
        other = self.labels(lam, not forward)
        x, neg = (self.root if forward else self.top), 0.0
        for t in range(self.k) if forward else range(self.k - 1, -1, -1):
            F, B = (x, other[t + 1]) if forward else (other[t], x)
            m0, m1 = self.marginals(F, B, t, lam[t])
            d = m1 - m0
            lam[t] += T[self.var[t]] - omega * d
            neg = neg + (-d).clamp(min=0.0)
            x = self.up(x, t, lam[t]) if forward else self.down(x, t, lam[t])
        return None if forward else (x[0] - omega * neg).sum()


class _Dual64:
    def __init__(self, g):
        self.n = g["n_vars"]
        dev = {k: torch.from_numpy(g[k]).to(DEV) for k in ("cost", "row_ptr", "col", "coef", "sense", "rhs")}
        self.cost = dev["cost"]
        col, coef, lens = dev["col"].long(), dev["coef"].long(), torch.diff(dev["row_ptr"])
        self.copies = torch.bincount(col, minlength=self.n)
        free = self.copies == 0
        self.const = float(self.cost[free].clamp(max=0.0).sum())
        self.inv = 1.0 / self.copies.clamp(min=1).double()
        mix = torch.from_numpy(np.random.default_rng(1).integers(1, 1 << 40, 4100)).to(DEV)
        self.groups, self.nnz = [], len(col)
        for k in torch.unique(lens).tolist():
            rows = torch.nonzero(lens == k).reshape(-1)
            slots = dev["row_ptr"][rows][:, None] + torch.arange(k, device=DEV)
            a = coef[slots]
            key = (a * mix[:k]).sum(1) + dev["sense"][rows].long() * mix[-1] + dev["rhs"][rows] * mix[-2]
            for u in torch.unique(key).tolist():
                sel = torch.nonzero(key == u).reshape(-1)
                j = int(rows[sel[0]])
                self.groups.append(_Rows64(a[sel[0]].tolist(), int(g["sense"][j]), int(g["rhs"][j]),
                                           slots[sel].t().contiguous(), col[slots[sel]].t().contiguous()))
        start = self.cost * self.inv
        self.lam = [start[r.var] for r in self.groups]
        self.T = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        self.lbs = []

    def _pass(self, omega, forward):
        parts = [r.sweep(lam, self.T, omega, forward) for r, lam in zip(self.groups, self.lam)]
        total = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for r, lam in zip(self.groups, self.lam):
            total.index_add_(0, r.var.reshape(-1), lam.reshape(-1))
        self.T = (self.cost - total) * self.inv
        return parts

    def iterate(self, iters, tol=0.0, omega=0.5, window=10, min_iters=20):
        for _ in range(iters):
            self._pass(omega, True)
            self.lbs.append(torch.stack(self._pass(omega, False)).sum())
            n = len(self.lbs)
            if tol > 0 and n >= min_iters and n > window:
                lb, before = float(self.lbs[-1]) + self.const, float(self.lbs[-1 - window]) + self.const
                if lb - before <= tol * max(abs(lb), 1.0):
                    break
        return len(self.lbs), float(self.lbs[-1]) + self.const

    def feasible_bound(self):
        return self.const + sum(float(r.labels(lam + self.T[r.var], False)[0][0].sum())
                                for r, lam in zip(self.groups, self.lam))

    def in_row_order(self, per_group):
        out = torch.empty(self.nnz, dtype=torch.float64, device=DEV)
        for r, x in zip(self.groups, per_group):
            out[r.slots] = x
        return out.cpu().numpy()

    def marginals(self):
        m0, m1 = [], []
        for r, lam in zip(self.groups, self.lam):
            F, B = r.labels(lam, True), r.labels(lam, False)
            got = [r.marginals(F[t], B[t + 1], t, lam[t]) for t in range(r.k)]
            m0.append(torch.stack([g[0] for g in got]))
            m1.append(torch.stack([g[1] for g in got]))
        return self.in_row_order(m0), self.in_row_order(m1)


def exact(case, seed):
    """Bounds, multipliers and min-marginals of Alg. 1 in 64 bits.  Rounded points are whole numbers that follow
    from the signs of 32-bit differences, so they have no value here."""
    op = case["op"]
    if op in ("batch", "serve"):
        return None
    if op == "reduce":
        v = prepare(case, seed)["values"].cpu().numpy()
        return {"sum": np.array([math.fsum(v) + 1.25])}
    d = _Dual64(_inputs(case, seed)[0])
    iters, lb = d.iterate(case["iters"], tol=1e-4 if op in ("solve", "from_host") else 0.0)
    if op == "iterate":
        return {"iters": None, "lb": lb, "lam": d.in_row_order(d.lam)}
    if op == "bound":
        return {"iters": None, "lb": lb, "lb_running": lb, "lb_feasible": d.feasible_bound()}
    if op == "read":
        m0, m1 = d.marginals()
        return {"lb": lb, "lb_feasible": d.feasible_bound(), "var": None, "row": None, "m0": m0, "m1": m1}
    return {"iters": None, "lb": lb, "status": None, "rounds": None, "x": None, "objective": None, "feasible": None}
