"""The product over C on both sides of the rule that chooses its kernel (the tile kernel or the row
groups): lattices and random graphs, short and long rows, the sizes at which the rule turns.

Bound, element by element: a row of k stored entries is k multiply-adds of rounded values and the
multiplier's term, (k + 4) u (|C| |X| + |a v| |X|) with u = 2^-24 for float arithmetic (the entries
of C and the weight are rounded to it as well) and 2^-53 for FP64.
"""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

import paper_2407_15049_gb300 as L
import workloads as W

pytestmark = pytest.mark.gpu

DT = {"fp64": (torch.float64, 2.0**-53), "fp32": (torch.float32, 2.0**-24), "bf16": (torch.bfloat16, 2.0**-24)}


def _graph(kind, n, deg):
    if kind == "torus":
        return W.maxcut_instance(n * n, W.torus_graph(n, 3, "pm1"))
    return W.maxcut_instance(n, W.er_graph(n, n * deg // 2, 3, "pm1"))


@pytest.mark.parametrize("kind,n,deg,r,prec", [
    ("torus", 560, 4, 20, "fp32"), ("torus", 560, 4, 16, "fp32"), ("torus", 900, 4, 13, "fp32"), ("torus", 300, 4, 20, "fp32"),
    ("torus", 560, 4, 20, "bf16"), ("torus", 560, 4, 5, "bf16"), ("torus", 300, 4, 12, "bf16"),
    ("er", 610000, 4, 20, "fp32"), ("er", 610000, 3, 20, "fp32"), ("er", 20011, 9, 27, "fp32"),
    ("er", 610000, 4, 20, "bf16"), ("er", 610000, 7, 19, "bf16"), ("er", 400003, 4, 32, "bf16"), ("er", 20011, 9, 27, "bf16"),
    ("er", 60013, 4, 16, "fp64"), ("er", 60013, 12, 16, "fp64"), ("er", 2003, 30, 20, "fp64"), ("er", 2003, 20, 20, "fp64"),
    ("er", 60013, 5, 64, "fp64"), ("er", 5003, 5, 64, "fp64"), ("er", 701, 300, 9, "fp64"), ("er", 701, 300, 9, "fp32"),
    ("er", 701, 300, 9, "bf16"), ("er", 1009, 5, 3, "fp64"), ("er", 1009, 5, 132, "fp64"),
])
def test_product_on_both_sides_of_the_rule(kind, n, deg, r, prec):
    dtype, u = DT[prec]
    inst = _graph(kind, n, deg)
    C = sp.csr_matrix((inst.val, inst.colind, inst.rowptr), shape=(inst.n, inst.n))
    gen = torch.Generator(device="cuda").manual_seed(7)
    X = torch.zeros((inst.n, L.padded_ld(r)), dtype=dtype, device="cuda")
    X[:, :r] = torch.randn(inst.n, r, generator=gen, dtype=torch.float64, device="cuda").to(dtype)
    v = torch.randn(inst.m, generator=gen, dtype=torch.float64, device="cuda")
    Xh, vh = X[:, :r].double().cpu().numpy(), v.cpu().numpy()
    w = np.zeros(inst.n)
    w[inst.row] = inst.aval * vh[inst.con]
    k = np.diff(inst.rowptr)[:, None] + 4
    ctx = L.lorads_create(inst)
    try:
        for mult in (None, v):
            out = torch.full(X.shape, float("nan"), dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
            L.lorads_spmm(ctx, X, mult, out, r=r)
            got = out.double().cpu().numpy()
            want, size = C @ Xh, abs(C) @ np.abs(Xh)
            if mult is not None:
                want = want - w[:, None] * Xh
                size = size + np.abs(w[:, None] * Xh)
            assert np.all(np.abs(got[:, :r] - want) <= k * u * size) and np.all(got[:, r:] == 0.0)
    finally:
        L.lorads_destroy(ctx)
