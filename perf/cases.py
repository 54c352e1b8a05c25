"""The calls that programs make of this library, at sizes from the smallest to the largest they use.

Each case is one public call (or the few calls that belong together) on a seeded
problem of the families the library is used for: the MaxCut SDP of a sparse graph
(X_ii = 1, C = -L/4) and the matrix-completion SDP (C = I, one constraint per
sampled entry).  Graphs, samples and factors are drawn on the GPU from the seed.

kinds
  spmm         out = (C - A*(v)) R, the gradient product
  cons         out_k = <A_k, U V^T>, the constraint map
  linesearch   the exact line-search coefficients a1..a4 and the step
  solve        the ALM solve from a given R0, a fixed slice of L-BFGS iterations, and its R and y
  admm_cg      one block step of the ADMM stage (conjugate gradients, a given number of steps)
  batch        many uneven instances in one persistent launch, a fixed slice of iterations, R and y of each
  gnn_train    one training step of the warm-start network on one graph
  gnn_predict  a starting factor for one graph from the network
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2407_15049_gb300 as L
from paper_2407_15049_gb300 import warmstart

DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16}
PREC = {"fp64": L.LORADS_FP64, "fp32": L.LORADS_FP32, "mixed": L.LORADS_MIXED}
FEATURES, HIDDEN, LAYERS, NORMALS = 16, 32, 3, 12
CG_TINY = 1e-12            # a CG stop that a few steps never reach: the step count is the case's


def listed():
    return [
        # The smallest call: a gradient product on a graph of a thousand vertices (per-call cost counts).
        dict(name="spmm er 1e3 fp64", kind="spmm", graph="er", n=1000, deg=8, r=10, prec="fp64", v=True),
        # The gradient product of the 1000 x 1000 torus workload in the float form.
        dict(name="spmm torus 1e6 fp32", kind="spmm", graph="torus", n=1000 * 1000, deg=4, r=20, prec="fp32", v=True),
        # The gradient product of the 50000 x 50000 matrix-completion workload (2.7e6 samples), bf16 rows.
        dict(name="spmm mc 1e5 bf16", kind="spmm", graph="mc", n=50000, n2=50000, r=22, prec="bf16", v=True),
        # The constraint map of a rectangular completion problem of odd sides and rank, U and V different.
        dict(name="cons mc 30011x50021 fp32", kind="cons", graph="mc", n=30011, n2=50021, r=17, prec="fp32", same=False),
        # An exact line search of the caller's own method on a sparse random graph, all in FP64.
        dict(name="linesearch er 1e6 fp64", kind="linesearch", graph="er", n=1000000, deg=4, r=20, prec="fp64"),
        # A small solve in FP64, the library's defaults: the host loop, the control kernels and launch latency.
        dict(name="solve er 1e3 fp64", kind="solve", graph="er", n=1000, deg=8, r=10, prec="fp64", mem=4, iters=60),
        # The main use: a large sparse MaxCut in the mixed form with two stored pairs, as the n = 1e7 workload runs it.
        dict(name="solve er 1e6 mixed", kind="solve", graph="er", n=1000000, deg=4, r=24, prec="mixed", mem=2, iters=24),
        # A matrix-completion solve (off-diagonal constraints) in the mixed form.
        dict(name="solve mc 4e4 mixed", kind="solve", graph="mc", n=20000, n2=20000, r=20, prec="mixed", mem=4, iters=40),
        # A block step of the ADMM stage of the torus workload.
        dict(name="admm_cg torus 1e6 fp32", kind="admm_cg", graph="torus", n=1000 * 1000, deg=4, r=20, prec="fp32", steps=10),
        # Serving: uneven small instances, MaxCut and completion, solved together.
        dict(name="batch 96 mixed", kind="batch", count=96, mix=1, nmin=200, nmax=8000, prec="mixed", iters=20),
        # Training the warm start on one of its larger graphs.
        dict(name="gnn_train er 3e4 bf16", kind="gnn_train", graph="er", n=30000, deg=4, r=24, act="bf16"),
        # A starting factor for a graph of a million vertices.
        dict(name="gnn_predict er 1e6 bf16", kind="gnn_predict", graph="er", n=1000000, deg=4, r=24, act="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, lo, hi):
    g = rng.choice(["er", "er", "torus"])
    n = _log_int(rng, lo, hi)
    if g == "torus":
        return dict(graph=g, n=max(4, int(round(math.sqrt(n)))) ** 2, deg=4)
    return dict(graph=g, n=n, deg=rng.randint(3, 12))


def _draw_mc(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    return dict(graph="mc", n=n, n2=max(lo, int(n * rng.uniform(0.5, 1.0))))


def _draw_any(rng, lo, hi, mc_lo, mc_hi):
    return _draw_mc(rng, mc_lo, mc_hi) if rng.random() < 0.35 else _draw_graph(rng, lo, hi)


def draw(rng):
    kind = rng.choice(["spmm", "cons", "linesearch", "solve", "solve", "admm_cg", "batch", "gnn_train", "gnn_predict"])
    r = rng.randint(4, 32)
    if kind == "spmm":
        return dict(kind=kind, **_draw_any(rng, 300, 1000000, 200, 50000), r=r,
                    prec=rng.choice(["fp64", "fp32", "bf16"]), v=rng.random() < 0.8)
    if kind == "cons":
        return dict(kind=kind, **_draw_any(rng, 300, 1000000, 200, 50000), r=r,
                    prec=rng.choice(["fp64", "fp32", "bf16"]), same=rng.random() < 0.5)
    if kind == "linesearch":
        return dict(kind=kind, **_draw_any(rng, 300, 1000000, 200, 50000), r=r, prec="fp64")
    if kind == "solve":
        c = _draw_any(rng, 300, 1000000, 200, 20000)
        rows = c["n"] + c.get("n2", 0)
        prec = rng.choice(["fp64", "mixed", "mixed"])
        return dict(kind=kind, **c, r=min(r, max(8, int(math.log2(rows)) + 4)), prec=prec, mem=rng.choice([2, 3, 4]),
                    iters=rng.randint(12, 30) if prec == "fp64" else rng.randint(12, 24))
    if kind == "admm_cg":
        return dict(kind=kind, **_draw_any(rng, 300, 1000000, 200, 20000), r=r, prec=rng.choice(["fp64", "fp32"]),
                    steps=rng.randint(4, 12))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(8, 96), mix=rng.randint(2, 10**6), nmin=200, nmax=_log_int(rng, 1000, 8000),
                    prec=rng.choice(["fp64", "mixed"]), iters=rng.randint(10, 20))
    if kind == "gnn_train":
        return dict(kind=kind, graph="er", n=_log_int(rng, 1000, 30000), deg=rng.randint(3, 8), r=r,
                    act=rng.choice(["bf16", "bf16", "fp32"]))
    return dict(kind=kind, graph="er", n=_log_int(rng, 1000, 1000000), deg=rng.randint(3, 8), r=r,
                act=rng.choice(["bf16", "bf16", "fp32"]))


# ------------------------------------------------------------------ problems
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda")


def _distinct(gen, total, count):
    """`count` distinct integers of [0, total), sorted."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < count:
        more = torch.randint(0, total, (int((count - keys.numel()) * 1.1) + 64,), generator=gen, device="cuda")
        keys = torch.unique(torch.cat([keys, more]))
    drop = torch.randperm(keys.numel(), generator=gen, device="cuda")[:count]
    return keys[torch.sort(drop).values]


def _edges(case, gen):
    n = case["n"]
    if case["graph"] == "torus":
        side = math.isqrt(n)
        idx = torch.arange(n, device="cuda").reshape(side, side)
        a = torch.cat([idx.reshape(-1), idx.reshape(-1)])
        c = torch.cat([idx.roll(-1, 1).reshape(-1), idx.roll(-1, 0).reshape(-1)])
        key = torch.unique(torch.minimum(a, c) * n + torch.maximum(a, c))
    else:
        # pairs i < j of the ER graph: distinct keys of the full square with the lower half folded up
        want = case["deg"] * n // 2
        key = torch.empty(0, dtype=torch.int64, device="cuda")
        while key.numel() < want:
            k = (want - key.numel()) + (want - key.numel()) // 20 + 64
            a = torch.randint(0, n, (k,), generator=gen, device="cuda")
            c = torch.randint(0, n, (k,), generator=gen, device="cuda")
            k2 = (torch.minimum(a, c) * n + torch.maximum(a, c))[a != c]
            key = torch.unique(torch.cat([key, k2]))
        keep = torch.randperm(key.numel(), generator=gen, device="cuda")[:want]
        key = key[torch.sort(keep).values]
    w = torch.randint(0, 2, (key.numel(),), generator=gen, device="cuda").double() * 2 - 1
    return key // n, key % n, w


def _host(t, dt):
    return t.to(dt).cpu().numpy()


def _instance(case, gen):
    """The SDP of the case in the library's exchange format (host arrays)."""
    if case["graph"] == "mc":
        n1, n2 = case["n"], case["n2"]
        n, m = n1 + n2, _samples(case)
        flat = _distinct(gen, n1 * n2, m)
        si, sj = flat // n2, flat % n2
        U, V = _randn(gen, n1, 3), _randn(gen, n2, 3)
        b = 2.0 * (U[si] * V[sj]).sum(1)
        rows = np.arange(n)
        return SimpleNamespace(n=n, rowptr=np.arange(n + 1), colind=rows.astype(np.int32), val=np.ones(n), m=m,
                               con=np.arange(m, dtype=np.int32), row=_host(si, torch.int32),
                               col=_host(sj + n1, torch.int32), aval=np.ones(m), b=_host(b, torch.float64))
    n = case["n"]
    i, j, w = _edges(case, gen)
    deg = torch.zeros(n, dtype=torch.float64, device="cuda")
    deg.index_add_(0, i, w).index_add_(0, j, w)              # sums of +-1: exact in any order
    d = torch.arange(n, device="cuda")
    key, order = torch.sort(torch.cat([i, j, d]) * n + torch.cat([j, i, d]))
    val = torch.cat([w / 4, w / 4, -deg / 4])[order]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    k = np.arange(n, dtype=np.int32)
    return SimpleNamespace(n=n, rowptr=_host(rowptr, torch.int64), colind=_host(key % n, torch.int32),
                           val=_host(val, torch.float64), m=n, con=k, row=k, col=k, aval=np.ones(n), b=np.ones(n))


def _samples(case):
    side = max(case["n"], case["n2"])
    return min(case["n"] * case["n2"] // 2, int(math.ceil(5 * side * math.log(side))))


def _factor(case, inst, gen, r):
    """A start as the solves take it: unit rows (MaxCut) or ||R||_F^2 = ||b||_1 / 2 (completion)."""
    R = _randn(gen, inst.n, r)
    if case["graph"] == "mc":
        return R * math.sqrt(0.5 * float(np.abs(inst.b).sum()) / float((R * R).sum()))
    return R / R.norm(dim=1, keepdim=True)


def _padded(R, dtype):
    out = torch.zeros(R.shape[0], L.padded_ld(R.shape[1]), dtype=dtype, device="cuda")
    out[:, :R.shape[1]] = R.to(dtype)
    return out


def _rho(inst):
    a = np.abs(inst.val[inst.val != 0])
    return 1.0 / float(a.mean()) if a.size else 1.0


class _Handle:
    """Keeps one library object and frees it with the state that holds it."""

    def __init__(self, obj, free):
        self.obj, self._free = obj, free

    def __del__(self):
        self._free(self.obj)


def _batch_cases(case):
    """About three MaxCut instances to one completion instance, sizes log-uniform; the mix is the case's."""
    u = np.random.default_rng(case["mix"]).random((case["count"], 3))
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
    out = []
    for a, b, c in u:
        n = int(round(math.exp(lo + (hi - lo) * b)))
        if a < 0.75:
            out.append(dict(graph="er", n=n, deg=3 + int(c * 10)))
        else:
            out.append(dict(graph="mc", n=max(100, n // 4), n2=max(100, n // 4)))
    return out


def _theta(gen, r):
    return (0.2 * _randn(gen, int(L.lorads_gnn_param_count(r)))).float()


def _inputs(case, seed):
    """Everything random of a case, drawn from the seed alone."""
    gen, kind = _gen(seed), case["kind"]
    s = SimpleNamespace()
    if kind == "batch":
        s.cases = _batch_cases(case)
        s.insts = [_instance(c, gen) for c in s.cases]
        s.R0 = [_factor(c, t, gen, max(1, math.ceil(math.log2(t.m)))) for c, t in zip(s.cases, s.insts)]
        return s
    s.inst = _instance(case, gen)
    if kind == "spmm":
        s.R = _padded(_factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
        s.v = _randn(gen, s.inst.m) if case["v"] else None
    elif kind == "cons":
        s.U = _padded(_factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
        s.V = s.U if case["same"] else _padded(_factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
    elif kind == "linesearch":
        s.R = _padded(_factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
        s.D = _padded(0.1 * _factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
        s.y, s.rho = 0.1 * _randn(gen, s.inst.m), _rho(s.inst)
    elif kind == "solve":
        s.R0 = _factor(case, s.inst, gen, case["r"])
    elif kind == "admm_cg":
        V = _factor(case, s.inst, gen, case["r"])
        s.V = _padded(V, DTYPE[case["prec"]])
        s.X = _padded(V + 0.01 * _factor(case, s.inst, gen, case["r"]), DTYPE[case["prec"]])
        s.y, s.rho = 0.1 * _randn(gen, s.inst.m), _rho(s.inst)
    else:
        s.theta = _theta(gen, case["r"])
        s.R = _factor(case, s.inst, gen, case["r"])
        s.feature_seed = int(seed) & 0xFFFF
    return s


def prepare(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    st = SimpleNamespace(kind=kind, case=case)
    if kind == "batch":
        b = L.lorads_batch_create(s.insts, L.default_params(prec=PREC[case["prec"]]),
                                  R0=[R.cpu().numpy() for R in s.R0])
        st.h, st.sizes = _Handle(b, L.lorads_batch_destroy), [(t.n, t.m) for t in s.insts]
        return st
    if kind.startswith("gnn"):
        st.graph = warmstart.device_graph(s.inst)
        st.net = warmstart.WarmStart(case["r"], act=case["act"], theta=s.theta.cpu().numpy())
        st.feature_seed = s.feature_seed
        if kind == "gnn_train":
            st.targets = warmstart.edge_targets(st.graph, _padded(s.R, torch.float64), case["r"])
        return st
    prm = L.default_params()
    if kind == "solve":
        prm = L.default_params(prec=PREC[case["prec"]], lbfgs_mem=case["mem"])
    st.h = _Handle(L.lorads_create(s.inst, prm), L.lorads_destroy)
    st.n, st.m = s.inst.n, s.inst.m
    for k in ("R", "v", "U", "V", "D", "y", "rho", "R0", "X"):
        if hasattr(s, k):
            setattr(st, k, getattr(s, k))
    return st


def _kept(x, case):
    """A solution as its user keeps it: the mixed form works in float, and its factor is rounded to
    cuts and entries in float."""
    return torch.as_tensor(x).float() if case["prec"] == "mixed" else x


def run(st):
    c, kind = st.case, st.kind
    if kind == "spmm":
        out = torch.empty(st.R.shape, dtype=torch.float64 if c["prec"] == "fp64" else torch.float32, device="cuda")
        L.lorads_spmm(st.h.obj, st.R, st.v, out, r=c["r"])
        return out
    if kind == "cons":
        out = torch.empty(st.m, dtype=torch.float64, device="cuda")
        L.lorads_constraint_eval(st.h.obj, st.U, st.V, out, r=c["r"])
        return out
    if kind == "linesearch":
        a, tau = L.lorads_linesearch_coeffs(st.h.obj, st.R, st.D, st.y, st.rho, r=c["r"])
        return {"a": a, "tau": tau}
    if kind == "solve":
        res = L.lorads_solve(st.h.obj, st.R0, max_total_inner=c["iters"])
        R, y = L.lorads_get_solution(st.h.obj, st.n, st.m)
        return {"R": _kept(R, c), "y": _kept(y, c), "inner": res["inner_iters"], "outer": res["outer_iters"]}
    if kind == "admm_cg":
        X = st.X.clone()                    # the block step overwrites its iterate
        steps = L.lorads_admm_cg(st.h.obj, st.V, X, st.y, st.rho, cg_rel=CG_TINY, cg_max=c["steps"], r=c["r"])
        return {"X": X, "steps": steps}
    if kind == "batch":
        res, _ = L.lorads_batch_solve(st.h.obj, c["count"], max_total_inner=c["iters"])
        sol = [L.lorads_batch_get_solution(st.h.obj, i, n, m) for i, (n, m) in enumerate(st.sizes)]
        return {"R": _kept(np.concatenate([R.ravel() for R, _ in sol]), c), "y": _kept(np.concatenate([y for _, y in sol]), c),
                "inner": np.array([r["inner_iters"] for r in res]), "outer": np.array([r["outer_iters"] for r in res])}
    if kind == "gnn_train":
        grad = torch.empty(int(L.lorads_gnn_param_count(c["r"])), dtype=torch.float32, device="cuda")
        st.net.train_step(st.graph, st.targets, 1e-3, st.feature_seed, grad_out=grad, want_loss=False)
        return grad
    return st.net.predict(st.graph, st.feature_seed)


# ------------------------------------------------------------------ what a pass cannot do without
def _sizes(case):
    """(n, nnz of C, m) of the case's problem; for an ER graph as it is asked for."""
    if case["graph"] == "mc":
        n = case["n"] + case["n2"]
        return n, n, _samples(case)
    n = case["n"]
    return n, n + 2 * (2 * n if case["graph"] == "torus" else case["deg"] * n // 2), n


def _iteration(case, r, wr, wd, mem):
    """Bytes and flops of one L-BFGS iteration: every array of the state read or written once."""
    n, nnz, m = _sizes(case)
    el = n * L.padded_ld(r)
    off = case["graph"] == "mc"
    by = el * ((2 + 2 * mem) * wd + 2 * wd + 4 * wr + 4 * wd) + nnz * (4 + wd) + 8 * (n + 1) + 28 * m
    return by, 2 * nnz * r + el * (4 * mem + 20) + (10 * m * r if off else 0)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # the instances of the mean size, as the seed draws them
        lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
        n = int((case["nmax"] - case["nmin"]) / (hi - lo))
        w8 = 8 if case["prec"] == "fp64" else 4
        parts = [_iteration(dict(graph="er", n=n, deg=8), max(1, math.ceil(math.log2(n))), 8, w8, 4)] * 3
        parts.append(_iteration(dict(graph="mc", n=n // 4, n2=n // 4), 12, 8, w8, 4))
        k = case["iters"] * case["count"] / 4
        return {"bytes": k * sum(p[0] for p in parts), "flops": k * sum(p[1] for p in parts)}
    n, nnz, m = _sizes(case)
    r = case["r"]
    el = n * L.padded_ld(r)
    if kind.startswith("gnn"):
        a = 2 if case["act"] == "bf16" else 4
        graph = nnz * 12 + 8 * n
        dense = 2 * n * (2 * HIDDEN * (FEATURES + 2 * HIDDEN) + HIDDEN * r) + 2 * nnz * (FEATURES + 2 * HIDDEN)
        if kind == "gnn_predict":
            return {"bytes": graph + 8 * el, "flops": dense}
        # a training step keeps each layer's input and message for its backward pass: written once, read once
        kept = 2 * n * a * (2 * FEATURES + 4 * HIDDEN + HIDDEN)
        return {"bytes": graph + nnz * 4 + kept, "flops": 3 * dense}
    w = {"fp64": 8, "fp32": 4, "bf16": 2, "mixed": 4}[case["prec"]]
    wv = max(w, 4)                                            # C's values: double, or float for the narrower rows
    off = m if case["graph"] == "mc" else 0
    cons = 28 * m                                             # row, column, coefficient and right-hand side or multiplier
    if kind == "spmm":
        return {"bytes": nnz * (4 + wv) + 8 * (n + 1) + el * (w + wv) + (cons if case["v"] else 0),
                "flops": 2 * nnz * r + (4 * off * r if case["v"] else 0)}
    if kind == "cons":
        return {"bytes": el * w * (1 if case["same"] else 2) + cons, "flops": 2 * m * r * (2 if off and not case["same"] else 1)}
    if kind == "linesearch":
        return {"bytes": nnz * (4 + wv) + 8 * (n + 1) + 2 * el * w + cons + 8 * m, "flops": 2 * nnz * r + 8 * m * r + 4 * el}
    if kind == "solve":
        by, fl = _iteration(case, r, 8, wv, case["mem"])
        return {"bytes": case["iters"] * by + 16 * n * r + 8 * m, "flops": case["iters"] * fl}
    # admm_cg: V read, r, p, X read and written and Q written and read in each step
    return {"bytes": case["steps"] * (el * w * 9 + cons) + nnz * (4 + wv) + 3 * el * w,
            "flops": case["steps"] * (el * 10 + 8 * m * r) + 2 * nnz * r}


# ------------------------------------------------------------------ the same in 64 bits
class _Sdp:
    """C, A and b of an instance as FP64 torch operators."""

    def __init__(self, inst):
        dev = dict(device="cuda")
        self.C = torch.sparse_csr_tensor(torch.as_tensor(inst.rowptr, **dev), torch.as_tensor(inst.colind, **dev).long(),
                                         torch.as_tensor(inst.val, **dev), (inst.n, inst.n))
        self.row, self.col = (torch.as_tensor(x, **dev).long() for x in (inst.row, inst.col))
        self.a, self.b = torch.as_tensor(inst.aval, **dev), torch.as_tensor(inst.b, **dev)
        self.off = bool((self.row != self.col).any())         # all constraints on the diagonal, or all off it

    def map(self, U, V):
        d = (U[self.row] * V[self.col]).sum(1)
        if self.off:
            d = d + (U[self.col] * V[self.row]).sum(1)
        return self.a * d

    def adj(self, v, X):
        w = (self.a * v)[:, None]
        out = torch.zeros_like(X).index_add_(0, self.row, w * X[self.col])
        return out.index_add_(0, self.col, w * X[self.row]) if self.off else out

    def slack(self, v, X):
        return self.C @ X - self.adj(v, X)

    def line(self, R, D, y, rho):
        """a1..a4 of the line search along D."""
        CD = self.C @ D
        q0 = self.b - self.map(R, R)
        q1, q2 = self.map(R, D) + self.map(D, R), self.map(D, D)
        w = y + rho * q0
        return [float(x) for x in (0.5 * rho * q2 @ q2, rho * q1 @ q2,
                                   (CD * D).sum() - w @ q2 + 0.5 * rho * q1 @ q1, 2 * (CD * R).sum() - w @ q1)]


def _step(a):
    """The positive root of the quartic's derivative with the lowest value (0: none lowers it)."""
    f = lambda t: (((a[0] * t + a[1]) * t + a[2]) * t + a[3]) * t  # noqa: E731
    best = 0.0
    for z in np.roots([4 * a[0], 3 * a[1], 2 * a[2], a[3]]):
        t = float(z.real)
        if t <= 0 or abs(z.imag) > 1e-6 * abs(t):
            continue
        for _ in range(3):                                    # Newton: the root to the last digits
            d2 = (12 * a[0] * t + 6 * a[1]) * t + 2 * a[2]
            t -= (((4 * a[0] * t + 3 * a[1]) * t + 2 * a[2]) * t + a[3]) / d2 if d2 else 0.0
        if t > 0 and f(t) < f(best):
            best = t
    return best


def _alm(inst, R, mem, iters, tol=1e-5):
    """`iters` L-BFGS iterations of the ALM solve in FP64: (R, y, iterations, outer steps)."""
    P = _Sdp(inst)
    binf, rho = float(P.b.abs().max()), _rho(inst)
    y = torch.zeros_like(P.b)
    dot = lambda u, v: float((u * v).sum())  # noqa: E731
    z = P.map(R, R) - P.b
    err, total, outer = float(z.norm()) / (1 + binf), 0, 0
    while True:
        S, Y = [], []
        G = 2 * P.slack(y - rho * z, R)
        g0, k = float(G.norm()), 0
        while True:
            if total >= iters:
                return R, y, total, outer
            thr = max(tol * (1 + binf), min(rho * float(z.norm()), 0.1 * g0))
            if float(G.norm()) <= thr or k >= 500:
                break
            D, al = -G, []
            for s, q in zip(reversed(S), reversed(Y)):
                al.append(dot(s, D) / dot(s, q))
                D = D - al[-1] * q
            if S:
                D = D * (dot(S[-1], Y[-1]) / dot(Y[-1], Y[-1]))
            for s, q, t in zip(S, Y, reversed(al)):
                D = D + (t - dot(q, D) / dot(s, q)) * s
            a = P.line(R, D, y, rho)
            a[3] = dot(G, D)
            tau = _step(a)
            k, total = k + 1, total + 1
            if tau <= 0:
                if not S:
                    break
                S, Y = [], []
                continue
            R = R + tau * D
            z = P.map(R, R) - P.b
            Gn = 2 * P.slack(y - rho * z, R)
            s, q = tau * D, Gn - G
            if dot(s, q) > 1e-16 * float(s.norm()) * float(q.norm()):
                S, Y = (S + [s])[-mem:], (Y + [q])[-mem:]
            else:
                S, Y = [], []
            G = Gn
        y = y - rho * z
        outer += 1
        e1 = float(z.norm()) / (1 + binf)
        obj, dual = float(((P.C @ R) * R).sum()), float(P.b @ y)
        if e1 <= tol and abs(obj - dual) <= tol * (1 + abs(obj) + abs(dual)):
            return R, y, total, outer
        if e1 > 0.25 * err and (k < 500 or e1 > err):
            rho = min(2 * rho, 1e12)
        err = e1


def _normals(n, seed):
    """The random node features: counter-based SplitMix64 and Box-Muller."""
    golden, mask = 0x9E3779B97F4A7C15, (1 << 64) - 1
    base = (seed ^ ((0x474E4E * golden) & mask)) & mask

    def out(k):
        z = np.uint64(base) + k * np.uint64(golden)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return (z ^ (z >> np.uint64(31))) >> np.uint64(11)

    with np.errstate(over="ignore"):
        e = np.arange(n * NORMALS, dtype=np.uint64) * np.uint64(2)
        u1 = (out(e + np.uint64(1)).astype(np.float64) + 1) / 2.0 ** 53
        u2 = out(e + np.uint64(2)).astype(np.float64) / 2.0 ** 53
    return torch.as_tensor((np.sqrt(-2 * np.log(u1)) * np.cos(2 * np.pi * u2)).reshape(n, NORMALS), device="cuda")


def _network(inst, theta, r, feature_seed):
    """(unit rows of the network, its edges) in FP64."""
    n = inst.n
    rp = torch.as_tensor(inst.rowptr, device="cuda")
    i = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    j, w = torch.as_tensor(inst.colind, device="cuda").long(), torch.as_tensor(inst.val, device="cuda")
    off = i != j
    total = lambda rows, x: torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, rows, x)  # noqa: E731
    diag, i, j, w = total(i[~off], w[~off]), i[off], j[off], w[off]
    s = total(i, w.abs())
    inv = torch.where(s > 0, 1 / s, torch.zeros_like(s))
    A = torch.sparse_coo_tensor(torch.stack([i, j]), w * inv[i], (n, n))
    x = torch.cat([torch.ones(n, 1, dtype=torch.float64, device="cuda"), (torch.log1p(total(i, torch.ones_like(w))) / 4)[:, None],
                   (total(i, w) * inv)[:, None], (diag * inv)[:, None], _normals(n, feature_seed)], 1)
    at, f = 0, FEATURES

    def take(*shape):
        nonlocal at
        at += math.prod(shape)
        return theta[at - math.prod(shape):at].reshape(shape)

    h = x
    for _ in range(LAYERS):
        Ws, Wn, b = take(HIDDEN, f), take(HIDDEN, f), take(HIDDEN)
        h, f = torch.relu(h @ Ws.T + torch.sparse.mm(A, h) @ Wn.T + b), HIDDEN
    Wo, bo = take(r, HIDDEN), take(r)
    o = h @ Wo.T + bo
    return o / o.norm(dim=1, keepdim=True), i, j


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "batch":
        got = [_alm(t, R, 4, case["iters"]) for t, R in zip(s.insts, s.R0)]
        return {"R": torch.cat([g[0].reshape(-1) for g in got]), "y": torch.cat([g[1] for g in got]), "inner": None, "outer": None}
    if kind.startswith("gnn"):
        theta = s.theta.double().requires_grad_(kind == "gnn_train")
        rows, i, j = _network(s.inst, theta, case["r"], s.feature_seed)
        if kind == "gnn_predict":
            return torch.nn.functional.pad(rows, (0, L.padded_ld(case["r"]) - case["r"]))
        up = i < j
        i, j = i[up], j[up]
        loss = (((rows[i] * rows[j]).sum(1) - (s.R[i] * s.R[j]).sum(1).float().double()) ** 2).mean()
        return torch.autograd.grad(loss, theta)[0]
    if kind == "solve":
        R, y, inner, outer = _alm(s.inst, s.R0, case["mem"], case["iters"])
        return {"R": R, "y": y, "inner": None, "outer": None}
    P = _Sdp(s.inst)
    if kind == "spmm":
        R = s.R.double()
        return P.slack(s.v, R) if case["v"] else P.C @ R
    if kind == "cons":
        return P.map(s.U.double(), s.V.double())
    if kind == "linesearch":
        a = P.line(s.R, s.D, s.y, s.rho)
        return {"a": np.array(a), "tau": _step(a)}
    V, X, rho = s.V.double(), s.X.double(), s.rho
    op = lambda Z: rho * (P.adj(P.map(Z, V), V) + Z)  # noqa: E731
    res = -(P.C @ V) + P.adj(s.y + rho * P.b, V) + rho * V - op(X)
    p, rr = res, float((res * res).sum())
    for _ in range(case["steps"]):
        q = op(p)
        al = rr / float((p * q).sum())
        X, res = X + al * p, res - al * q
        new = float((res * res).sum())
        p, rr = res + (new / rr) * p, new
    return {"X": X, "steps": None}
