"""The work that programs on this library have it do, as cases that can be timed and compared.

A case is a dict of plain values. `prepare` makes what a caller holds before a call: node boxes, split
counts or points of the seed, and the problem handle. Handles are kept per tape and options, as a
branch-and-bound program keeps one for its whole search. `run` is one call of a public entry point.
`exact` is the same result in plain torch float64: intervals by endpoint formulas, rounded to nearest.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2507_20769_gb300 import autograd, ivb
from paper_2507_20769_gb300 import workloads as W

DEV = "cuda:0"


# ------------------------------------------------------------------ cases

def _case(name, kind, tape, **kw):
    c = {"name": name, "kind": kind, "tape": tape, "nodes": 1, "target": 256, "target_max": 0, "grad": "adjoint",
         "form": "mvf", "filter": 0, "specialize": -1, "host": False, "first": 0, "count": 0}
    c.update(kw)
    return c


def listed():
    return [
        # one node of a two-variable problem, host arrays, default options: the first call of any new user, and
        # the shape of a search that bounds node by node
        _case("tiny_node", "bound", "config 1", target=256, specialize=0, host=True),
        # children of one small branch-and-bound iteration on the same problem: launches and latency
        _case("tiny_batch", "bound", "config 1", nodes=31, target=256),
        # the plain path: forward tangents, default options, 16^4 subdomains per node
        _case("plain_forward", "bound", "config 2", nodes=12, target=65536, grad="forward", specialize=0),
        # an iteration of the four-variable constrained problem, adjoint gradients, the library's kernel choice
        _case("plain_adjoint", "bound", "config 2", nodes=64, target=65536),
        # uneven nodes with the default options (tape interpreter, adjoint)
        _case("uneven_default", "bound", "config 3", nodes=48, target=256, target_max=8192, specialize=0),
        # a full batch of 256 uneven nodes, constraints, the library's kernel choice
        _case("uneven_batch", "bound", "config 3", nodes=256, target=1024, target_max=65536),
        # one iteration of a converging search: meet of both forms, certainly infeasible subdomains skipped
        _case("search_iteration", "bound", "config 3", nodes=61, target=8192, form="mvf_nie", filter=1),
        # sixteen variables, one node, about 2^20 subdomains
        _case("wide_node", "bound", "config 4", target=1 << 20),
        # the full-scale problem: eleven outputs of 1000 entries, 2^18 subdomains per node
        _case("full_scale", "bound", "config 5", nodes=6, target=1 << 18),
        # enclosures, point values and gradients of a range of one node's subdomains, for a caller that
        # inspects or plots them
        _case("enclose_range", "enclose", "config 3", target=1 << 17, first=1001, count=50_003, specialize=0),
        # value and gradient at many points through autograd, forward and backward (multistart descent)
        _case("point_gradients", "points", "config 4", nodes=100_003, specialize=0),
        # a whole search on a rational problem with one constraint, propagation on the host
        _case("whole_search", "search", "rational 3 40 1 2 4242", nodes=16, target=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MOST_OPS = 4.0e10      # directed endpoint operations of one drawn case at most (the largest listed one has 9.3e10)


def draw(rng):
    kind = rng.choice(["bound"] * 6 + ["noalloc", "enclose", "points", "search"])
    while True:
        if kind == "search":
            tape = "rational %d %d %d 2 %d" % (rng.randint(2, 4), _log_int(rng, 20, 60), rng.randint(0, 2), rng.randrange(10 ** 6))
            return _unnamed(_case("", kind, tape, nodes=rng.randint(1, 32), target=_log_int(rng, 64, 2048),
                                  specialize=rng.choice([0, -1])))
        if rng.random() < 0.5:
            tape = "config %d" % rng.randint(1, 3 if kind == "noalloc" else 5)
        else:
            tape = "random %d %d %d %d %d" % (rng.randint(2, 16), _log_int(rng, 24, 1000), rng.randint(0, 10),
                                              rng.choice([2, 5, 10]), rng.randrange(10 ** 6))
        c = _case("", kind, tape, nodes=_log_int(rng, 1, 256), target=_log_int(rng, 200, 1 << 18),
                  grad=rng.choice(["adjoint", "adjoint", "adjoint", "forward"]),
                  form=rng.choice(["mvf", "mvf", "mvf_nie", "nie"]), filter=rng.choice([0, 0, 1]),
                  specialize=rng.choice([0, -1, -1]), host=rng.random() < 0.25)
        if kind == "noalloc":
            if tape.startswith("random") and int(tape.split()[2]) > 250:
                continue       # a thread's frame has to fit in shared memory
            c["host"] = False
        if kind == "enclose":
            c.update(nodes=1, count=_log_int(rng, 100, 100_000), first=rng.randint(0, 1000), form="mvf", filter=0)
            c["target"] = 4 * (c["count"] + c["first"])
        if kind == "points":
            c.update(nodes=_log_int(rng, 10, 1_000_000), grad="adjoint", form="mvf", filter=0, host=False)
        if c["grad"] == "forward":
            c["specialize"] = 0
        if work(c)["flops"] <= MOST_OPS and (kind != "enclose" or _tape(tape).n_vars <= 16):
            return _unnamed(c)


def _unnamed(c):
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _tape(spec):
    kind, *num = spec.split()
    num = [int(v) for v in num]
    if kind == "config":
        return W.config_tape(num[0])
    n, K, m, half, seed = num
    ops = W.OPS_RATIONAL if kind == "rational" else W.OPS_ALL
    return W.random_problem(n, max(K, n + 8), m, ops, [[-half, half]] * n, seed, spec)


@functools.lru_cache(maxsize=None)
def _problem(tape, grad, form, filt, specialize):
    return ivb.Problem(_tape(tape), grad_mode=grad, form=form, filter=filt, specialize=specialize)


def _nodes(case, seed):
    """node boxes [k, n, 2] and split counts [k, n]: bisections of a tightened root box (about half of its ends
    moved inwards, as propagation leaves them), or nodes of uneven widths and subdomain counts"""
    t = _tape(case["tape"])
    k, root = case["nodes"], t.root_box.copy()
    rng = np.random.default_rng(seed)
    if case["target_max"]:
        lo, hi = (int(math.log2(case[q])) for q in ("target", "target_max"))
        boxes, targets = W.uneven_nodes(t.n_vars, k, root, seed, log2_s=(lo, hi))
    else:
        w = root[:, 1] - root[:, 0]
        move = rng.uniform(0.0, 0.1, root.shape) * (rng.random(root.shape) < 0.5)
        move[0, 0] = 0.05 + 0.05 * rng.random()
        root[:, 0] += w * move[:, 0]
        root[:, 1] -= w * move[:, 1]
        boxes, targets = W.bisection_frontier(root, k, seed), np.full(k, case["target"])
    ref = t.root_box[:, 1] - t.root_box[:, 0]
    splits = np.stack([ivb.ivb_pick_splits(b, int(g), "adaptive", ref) for b, g in zip(boxes, targets)])
    return np.ascontiguousarray(boxes), np.ascontiguousarray(splits, dtype=np.int32)


def prepare(case, seed):
    t = _tape(case["tape"])
    p = _problem(case["tape"], case["grad"], case["form"], case["filter"], case["specialize"])
    s = {"case": case, "p": p}
    if case["kind"] == "points":
        lo, hi = (torch.from_numpy(np.ascontiguousarray(t.root_box[:, q])).to(DEV) for q in (0, 1))
        g = torch.Generator(device=DEV).manual_seed(seed)
        u = torch.rand((case["nodes"], t.n_vars), dtype=torch.float64, device=DEV, generator=g)
        s["x"] = (lo + (hi - lo) * u).requires_grad_()
        s["grad_f"] = torch.randn((case["nodes"], t.n_out), dtype=torch.float64, device=DEV, generator=g)
        return s
    s["boxes"], s["splits"] = _nodes(case if case["kind"] != "search" else dict(case, nodes=1), seed)
    if case["kind"] != "search" and not case["host"]:
        s["boxes"], s["splits"] = (torch.from_numpy(v).to(DEV) for v in (s["boxes"], s["splits"]))
    if case["kind"] == "noalloc":
        s["lb"] = torch.empty(case["nodes"], dtype=torch.float64, device=DEV)
        s["infeasible"] = torch.empty(case["nodes"], dtype=torch.uint8, device=DEV)
    return s


# -------------------------------------------------------------------- run

def run(s):
    c, p = s["case"], s["p"]
    if c["kind"] == "bound":
        return p.bound_nodes_ex(s["boxes"], s["splits"], want_hull=True)
    if c["kind"] == "noalloc":
        return p.bound_nodes_noalloc(s["boxes"], s["splits"], s["lb"], s["infeasible"])
    if c["kind"] == "enclose":
        return p.enclose(s["boxes"][0], s["splits"][0], first=c["first"], count=c["count"], want_fc=True, want_g=True)
    if c["kind"] == "points":
        f = autograd.point_values(p, s["x"])
        (g,) = torch.autograd.grad(f, s["x"], s["grad_f"])
        return f.detach(), g
    r = p.bnb_solve(s["boxes"][0], splits=s["splits"][0], batch=c["nodes"], eps_rel=1e-3, max_nodes=3000, propagate=2)
    return {k: r[k] for k in ("lb", "ub", "converged", "nodes", "subdomains")}


def _subdomains(case):
    """about: what the adaptive picker gets within the targets"""
    if case["kind"] == "enclose":
        return case["count"]
    if case["target_max"]:
        lo, hi = (int(math.log2(case[q])) for q in ("target", "target_max"))
        return case["nodes"] * sum(1 << q for q in range(lo, hi + 1)) / (hi - lo + 1)
    return case["nodes"] * case["target"]


def work(case):
    """bytes of the arrays read and written; flops: directed endpoint operations of the canonical formulas (value
    sweep on [c,c] and on X, tangents or adjoints, Mean Value Form), one per interval end"""
    t = _tape(case["tape"])
    n, m = t.n_vars, t.n_out
    const = t.op == W.OP_CONST
    value = grad = 0.0
    for op, a, b in zip(t.op.tolist(), t.a.tolist(), t.b.tolist()):
        if op in (W.OP_VAR, W.OP_CONST, W.OP_NEG):
            continue
        value += 2
        parts = 2 * ((not const[a]) + (op in W.BINARY and not const[b]))
        grad += parts + {W.OP_DIV: 4, W.OP_SQRT: 2, W.OP_LOG: 2}.get(op, 0)
    if case["kind"] == "points":
        k = case["nodes"]
        return {"bytes": 8.0 * k * (n + 2 * m + n), "flops": k * (value + grad) / 2}
    subs = _subdomains(case)
    if case["form"] == "nie":
        grad = 0.0
    per = 2 * value + grad * (n if case["grad"] == "forward" else 1) + (4 * n * m if grad else 0) + 6 * n
    if case["kind"] == "search":
        return {"bytes": 20.0 * n + 40, "flops": 100 * subs * per}      # some hundred nodes per search
    k = case["nodes"]
    out = subs * m * (4 + 2 * n) * 8 if case["kind"] == "enclose" else k * (17.0 + 16 * m) if case["kind"] == "bound" else 9.0 * k
    return {"bytes": 20.0 * n * k + out, "flops": float(subs * per)}


# ------------------------------------------------- the same in plain torch

INF = math.inf


def _add(x, y):
    return x[0] + y[0], x[1] + y[1]


def _sub(x, y):
    return x[0] - y[1], x[1] - y[0]


def _mul(x, y):
    p = [torch.nan_to_num(torch.as_tensor(a * b), nan=0.0, posinf=INF, neginf=-INF) for a in x for b in y]
    return torch.minimum(torch.minimum(p[0], p[1]), torch.minimum(p[2], p[3])), \
        torch.maximum(torch.maximum(p[0], p[1]), torch.maximum(p[2], p[3]))


def _where(ok, x):
    return torch.where(ok, x[0], -INF), torch.where(ok, x[1], INF)


def _recip(x):
    return _where((x[0] > 0) | (x[1] < 0), (1.0 / x[1], 1.0 / x[0]))


def _value(op, x, y):
    if op == W.OP_ADD:
        return _add(x, y)
    if op == W.OP_SUB:
        return _sub(x, y)
    if op == W.OP_MUL:
        return _mul(x, y)
    if op == W.OP_DIV:
        q = [a / b for a in x for b in y]
        lo = torch.minimum(torch.minimum(q[0], q[1]), torch.minimum(q[2], q[3]))
        hi = torch.maximum(torch.maximum(q[0], q[1]), torch.maximum(q[2], q[3]))
        return _where((y[0] > 0) | (y[1] < 0), (lo, hi))
    if op == W.OP_SQR:
        a, b = x[0].abs(), x[1].abs()
        return torch.where((x[0] <= 0) & (x[1] >= 0), 0.0, torch.minimum(a, b)) ** 2, torch.maximum(a, b) ** 2
    if op == W.OP_SQRT:
        return _where(x[0] >= 0, (x[0].sqrt(), x[1].sqrt()))
    if op == W.OP_EXP:
        return x[0].exp(), x[1].exp()
    if op == W.OP_LOG:
        return _where(x[0] > 0, (x[0].log(), x[1].log()))
    return -x[1], -x[0]


def _values(t, X):
    v = []
    for op, a, b, c in zip(t.op.tolist(), t.a.tolist(), t.b.tolist(), t.c.tolist()):
        if op == W.OP_VAR:
            v.append(X[a])
        elif op == W.OP_CONST:
            k = torch.full_like(X[0][0], c)
            v.append((k, k))
        else:
            v.append(_value(op, v[a], v[b]))
    return v


def _partials(op, x, y, v):
    """d v / d a and d v / d b as interval factors, a quotient's second one as (factor, factor)"""
    if op == W.OP_MUL:
        return y, x
    if op == W.OP_SQR:
        return (2 * x[0], 2 * x[1]), None
    if op == W.OP_SQRT:
        r = (2 * v[0], 2 * v[1])
        return _where(r[0] > 0, _recip(r)), None
    if op == W.OP_EXP:
        return v, None
    if op == W.OP_LOG:
        return _where(x[0] > 0, _recip(x)), None
    return None, None


def _adjoint(t, v, out, n):
    zero = (torch.zeros_like(v[0][0]),) * 2
    bar = {out: (torch.ones_like(v[0][0]),) * 2}

    def add(i, w):
        if t.op[i] != W.OP_CONST:
            bar[i] = _add(bar[i], w) if i in bar else w

    for i in range(out, n - 1, -1):
        if i not in bar:
            continue
        w, op, a, b = bar[i], int(t.op[i]), int(t.a[i]), int(t.b[i])
        if op in (W.OP_VAR, W.OP_CONST):
            continue
        del bar[i]
        if op == W.OP_ADD:
            add(a, w)
            add(b, w)
        elif op == W.OP_SUB:
            add(a, w)
            add(b, (-w[1], -w[0]))
        elif op == W.OP_NEG:
            add(a, (-w[1], -w[0]))
        elif op == W.OP_DIV:
            r = _recip(v[b])
            add(a, _mul(w, r))
            q = _mul(w, v[i])
            add(b, _mul((-q[1], -q[0]), r))
        else:
            da, db = _partials(op, v[a], v[b], v[i])
            add(a, _mul(w, da))
            if db is not None:
                add(b, _mul(w, db))
    return [bar.get(i, zero) for i in range(n)]


def _tangents(t, v, n):
    """per entry its n tangent intervals as ([n, m], [n, m]); None where they are zero"""
    d = []
    for i, (op, a, b) in enumerate(zip(t.op.tolist(), t.a.tolist(), t.b.tolist())):
        if op == W.OP_CONST:
            d.append(None)
            continue
        if op == W.OP_VAR:
            e = torch.zeros((n,) + v[0][0].shape, dtype=torch.float64, device=v[0][0].device)
            e[a] = 1.0
            d.append((e, e))
            continue
        da, db = d[a], d[b] if op in W.BINARY else None
        if op in (W.OP_ADD, W.OP_SUB):
            nb = None if db is None else db if op == W.OP_ADD else (-db[1], -db[0])
            d.append(nb if da is None else da if nb is None else _add(da, nb))
        elif op == W.OP_NEG:
            d.append(None if da is None else (-da[1], -da[0]))
        elif op == W.OP_DIV:
            q = None if db is None else _mul((-v[i][1], -v[i][0]), db)
            s = q if da is None else da if q is None else _add(da, q)
            d.append(None if s is None else _mul(s, _recip(v[b])))
        else:
            fa, fb = _partials(op, v[a], v[b], v[i])
            pa = None if da is None else _mul(fa, da)
            pb = None if db is None or fb is None else _mul(fb, db)
            d.append(pb if pa is None else pa if pb is None else _add(pa, pb))
    return d


def _enclose(case, boxes, splits, node, k):
    """F, f(c) and G of every output on subdomains k of nodes `node`"""
    t = _tape(case["tape"])
    n = t.n_vars
    X, C = [], []
    for i in range(n):
        lo, hi, N = boxes[node, i, 0], boxes[node, i, 1], splits[node, i].long()
        j, k = k % N, k // N
        h = (hi - lo) / N
        e0 = torch.where(j > 0, torch.minimum(torch.maximum(lo + j * h, lo), hi), lo)
        e1 = torch.where(j + 1 < N, torch.minimum(torch.maximum(lo + (j + 1) * h, lo), hi), hi)
        c = (e0 + e1) * 0.5
        X.append((e0, e1))
        C.append((c, c))
    fc = _values(t, C)
    v = _values(t, X)
    d = _tangents(t, v, n) if case["grad"] == "forward" and case["form"] != "nie" else None
    F, Fc, G = [], [], []
    for o in t.out_idx.tolist():
        f, g = fc[o], []
        if case["form"] != "nie":
            if d is None:
                g = _adjoint(t, v, o, n)
            else:
                z = torch.zeros_like(v[0][0])
                g = [(z, z) if d[o] is None else (d[o][0][i], d[o][1][i]) for i in range(n)]
            for i in range(n):
                f = _add(f, _mul(g[i], (X[i][0] - C[i][0], X[i][1] - C[i][0])))
            if case["form"] == "mvf_nie":
                f = torch.maximum(f[0], v[o][0]), torch.minimum(f[1], v[o][1])
        else:
            f = v[o]
        F.append(f)
        Fc.append(fc[o])
        G.append(g)
    return F, Fc, G


def _points(case, seed):
    t = _tape(case["tape"])
    s = prepare(case, seed)
    x = s["x"].detach().clone().requires_grad_()
    v = []
    for op, a, b, c in zip(t.op.tolist(), t.a.tolist(), t.b.tolist(), t.c.tolist()):
        v.append(x[:, a] if op == W.OP_VAR else torch.full_like(x[:, 0], c) if op == W.OP_CONST else
                 v[a] + v[b] if op == W.OP_ADD else v[a] - v[b] if op == W.OP_SUB else
                 v[a] * v[b] if op == W.OP_MUL else v[a] / v[b] if op == W.OP_DIV else
                 v[a] * v[a] if op == W.OP_SQR else v[a].sqrt() if op == W.OP_SQRT else
                 v[a].exp() if op == W.OP_EXP else v[a].log() if op == W.OP_LOG else -v[a])
    f = torch.stack([v[o] for o in t.out_idx.tolist()], 1)
    (g,) = torch.autograd.grad(f, x, s["grad_f"])
    return f.detach(), g


def exact(case, seed):
    t = _tape(case["tape"])
    if case["kind"] == "search" or (case["kind"] != "points" and work(case)["flops"] > 2.5e10):
        return None
    if case["kind"] == "points":
        return _points(case, seed) if case["nodes"] * t.n_ops < 4e8 else None
    boxes, splits = (torch.from_numpy(v).to(DEV) for v in _nodes(case, seed))
    if case["kind"] == "enclose":
        k = torch.arange(case["first"], case["first"] + case["count"], device=DEV)
        F, Fc, G = _enclose(case, boxes, splits, torch.zeros_like(k), k)
        both = lambda f: torch.stack([f[0].expand(k.shape), f[1].expand(k.shape)], 1)  # noqa: E731
        return (torch.stack([both(f) for f in F], 1), torch.stack([both(f) for f in Fc], 1),
                torch.stack([torch.stack([both(g) for g in G1], 1) for G1 in G], 1))
    kn, m = case["nodes"], t.n_out
    per = splits.long().prod(1)
    off = torch.cat([torch.zeros(1, dtype=torch.long, device=DEV), per.cumsum(0)])
    total = int(off[-1])
    ends = t.n_ops * 2 * (t.n_vars + 1 if case["grad"] == "forward" else 2)
    step = max(1 << 12, min(1 << 20, int(2e10 / (8 * ends))))
    if case["kind"] != "points" and total / step * t.n_ops * m > 4e5:
        return None
    obj = t.out_kind.tolist().index(W.KIND_OBJ)
    minlo = torch.full((kn, m), INF, dtype=torch.float64, device=DEV)
    maxhi = -minlo
    lb, ub = (torch.full((kn,), INF, dtype=torch.float64, device=DEV) for _ in range(2))
    for k0 in range(0, total, step):
        g = torch.arange(k0, min(total, k0 + step), device=DEV)
        node = torch.searchsorted(off, g, right=True) - 1
        F, Fc, _ = _enclose(case, boxes, splits, node, g - off[node])
        out = torch.zeros_like(g, dtype=torch.bool)
        ok = torch.ones_like(out)
        for o, kind in enumerate(t.out_kind.tolist()):
            lo, hi = (q.expand(g.shape) for q in F[o])
            minlo[:, o].scatter_reduce_(0, node, lo, "amin")
            maxhi[:, o].scatter_reduce_(0, node, hi, "amax")
            if kind == W.KIND_INEQ:
                out |= lo > 0
                ok &= Fc[o][1] <= 0
        lo = F[obj][0].expand(g.shape)
        lb.scatter_reduce_(0, node, torch.where(out, INF, lo) if case["filter"] else lo, "amin")
        ub.scatter_reduce_(0, node, torch.where(ok, Fc[obj][1].expand(g.shape), INF), "amin")
    if case["kind"] == "noalloc":
        return lb, None
    return {"lb": lb, "infeasible": None, "ub": ub, "minlo": minlo, "maxhi": maxhi}
