"""Sums of the line search and of the objective that a shorter accumulation would lose.

Each input is chosen so that the value is exact in the arithmetic that the pass states, and
not in a cheaper one, so the expected value is exact and has no tolerance.
"""
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
