"""Sums of the line search and of the objective that a shorter accumulation would lose.

Each input is chosen so that the value is exact in the arithmetic that the pass states, and
not in a cheaper one, so the expected value is exact and has no tolerance.
"""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_2407_15049_gb300 as L
import workloads as W

pytestmark = pytest.mark.gpu


def _one_offdiagonal(n, i, j):
    """C = one stored entry of the last row (where every factor here is 0), one constraint X_ij = 0."""
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[n] = 1
    return W.SDPInstance(n=n, rowptr=rowptr, colind=np.array([n - 1], np.int32), val=np.array([1.0]), m=1,
                         con=np.array([0], np.int32), row=np.array([i], np.int32), col=np.array([j], np.int32),
                         aval=np.array([1.0]), b=np.array([0.0]), kind="generic")


@pytest.mark.parametrize("ld", [4, 8, 20, 64, 128, 132])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("swap", [False, True])
def test_q1_adds_its_two_dots_beyond_float(ld, dtype, swap):
    """q1 = 2 (r_i.d_j + d_i.r_j) with the dots 2^24 and 1: each is exact in float, their sum is
    not.  With rho = 0 and C = 0 on these rows, a4 = -y q1."""
    n, i, j = 9, 2, 5
    inst = _one_offdiagonal(n, i, j)
    R = torch.zeros((n, ld), dtype=dtype, device="cuda")
    D = torch.zeros((n, ld), dtype=dtype, device="cuda")
    big, one = (R, D) if not swap else (D, R)
    big[i, 0], one[j, 0] = 4096.0, 4096.0
    one[i, ld - 1], big[j, ld - 1] = 1.0, 1.0
    ctx = L.lorads_create(inst)
    try:
        a, _ = L.lorads_linesearch_coeffs(ctx, R, D, torch.full((1,), 1.0, dtype=torch.float64, device="cuda"), 0.0)
    finally:
        L.lorads_destroy(ctx)
    assert a[3] == -2.0 * (2.0**24 + 1.0)
    assert a[0] == a[1] == a[2] == 0.0


@pytest.mark.parametrize("ld", [16, 20, 24, 32, 64, 128, 256])
@pytest.mark.parametrize("dtype,big", [(torch.float32, 4096.0), (torch.bfloat16, 4096.0), (torch.float64, 2.0**27)])
def test_row_sums_add_as_a_tree(ld, dtype, big):
    """r_i.d_i of a diagonal constraint, with big^2, 1, -big^2 in the first, second and (L/2)-th group of
    four elements, L the lanes of a row: the tree over the lanes pairs the first with the third and
    keeps the 1, a chain over them loses it."""
    n, i = 9, 4
    lanes = 1
    while lanes < min(ld // 4, 32):
        lanes *= 2
    inst = _one_offdiagonal(n, i, i)
    R = torch.zeros((n, ld), dtype=dtype, device="cuda")
    D = torch.zeros((n, ld), dtype=dtype, device="cuda")
    for unit, r, d in ((0, big, big), (1, 1.0, 1.0), (lanes // 2, big, -big)):
        R[i, 4 * unit], D[i, 4 * unit] = r, d
    ctx = L.lorads_create(inst)
    try:
        a, _ = L.lorads_linesearch_coeffs(ctx, R, D, torch.full((1,), 1.0, dtype=torch.float64, device="cuda"), 0.0)
    finally:
        L.lorads_destroy(ctx)
    assert a[3] == -2.0


def test_fp64_line_search_sums_its_rows_before_the_walk():
    """C = I and every four elements of R = D with the squares e, e, e, 1, e = 2^-48.  A thread walks 128
    rows, so its sum grows to 128 and e is half an ulp of it or less from 32 on: added one by one
    they are lost (8e-15 of the sum).  Added a tile at a time the sum takes at most 128 additions of
    at least one row, 22 for tiles of six, each off by half an ulp of 128 at most: 1.2e-15, and the
    folds over the blocks round a dozen times (1.3e-15)."""
    ld, e = 128, 2.0**-48
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 4
    n = 128 * warps
    inst = W.SDPInstance(n=n, rowptr=np.arange(n + 1, dtype=np.int64), colind=np.arange(n, dtype=np.int32),
                         val=np.ones(n), m=1, con=np.array([0], np.int32), row=np.array([0], np.int32),
                         col=np.array([0], np.int32), aval=np.array([1.0]), b=np.array([1.0]), kind="generic")
    row = torch.tensor([2.0**-24] * 3 + [1.0], dtype=torch.float64, device="cuda").repeat(ld // 4)
    R = row.repeat(n, 1).contiguous()
    ctx = L.lorads_create(inst)
    try:
        a, _ = L.lorads_linesearch_coeffs(ctx, R, R.clone(), torch.zeros(1, dtype=torch.float64, device="cuda"), 0.0)
    finally:
        L.lorads_destroy(ctx)
    want = n * (ld // 4) * (1 + 3 * Fraction(e))
    assert abs(Fraction(float(a[2])) - want) <= Fraction(2.5e-15) * want
    assert abs(Fraction(float(a[3])) - 2 * want) <= Fraction(2.5e-15) * 2 * want


def _f32(q: Fraction) -> Fraction:
    """q rounded to the nearest float (ties to even; the values here are normal)."""
    if q == 0:
        return q
    e = math.floor(math.log2(abs(q)))
    while abs(q) >= Fraction(2) ** (e + 1):
        e += 1
    while abs(q) < Fraction(2) ** e:
        e -= 1
    ulp = Fraction(2) ** (e - 23)
    return Fraction(round(q / ulp)) * ulp


def _two_sum(a, b):
    s = _f32(a + b)
    return s, a + b - s


def _dw_mul(x, y):
    """DWTimesDW with fused multiply-adds (Joldes, Muller, Popescu 2017)."""
    ch = _f32(x[0] * y[0])
    cl1 = x[0] * y[0] - ch
    cl2 = _f32(x[1] * y[0] + _f32(x[0] * y[1] + _f32(x[1] * y[1])))
    return _two_sum(ch, _f32(cl1 + cl2))


def _dw_add(x, y):
    """AccurateDWPlusDW of the same paper."""
    sh, sl = _two_sum(x[0], y[0])
    th, tl = _two_sum(x[1], y[1])
    vh, vl = _two_sum(sh, _f32(sl + th))
    return _two_sum(vh, _f32(tl + vl))


def test_double_float_dots_are_double_word_multiply_adds():
    """The objective at the start of a double-float solve, for a C of one stored diagonal entry 1 and rows
    of four elements: one lane's dot, the double-word multiply-add of its elements in turn."""
    n = 5
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[3:] = 1
    inst = W.SDPInstance(n=n, rowptr=rowptr, colind=np.array([2], np.int32), val=np.array([1.0]), m=n,
                         con=np.arange(n, dtype=np.int32), row=np.arange(n, dtype=np.int32),
                         col=np.arange(n, dtype=np.int32), aval=np.ones(n), b=np.ones(n), kind="generic")
    ctx = L.lorads_create(inst, L.default_params(prec=L.LORADS_DF64, max_outer=1, tol=1e-300))
    rng = np.random.default_rng(11)
    try:
        for _ in range(40):
            R0 = rng.standard_normal((n, 4))
            got = L.lorads_solve(ctx, R0, max_total_inner=1)["primal_obj"]
            acc = (Fraction(0), Fraction(0))
            for v in R0[2]:
                hi = Fraction(float(np.float32(v)))
                x = (hi, _f32(Fraction(float(v)) - hi))
                acc = _dw_add(_dw_mul(x, x), acc)
            assert got == float(acc[0] + acc[1])
    finally:
        L.lorads_destroy(ctx)
