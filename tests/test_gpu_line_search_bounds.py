"""The line search's coefficients within the rounding of each constraint's own dots.

Every quantity carries the bound of the operations that form it: a dot of r products in lanes of
4 c elements and a tree of 5 levels has the error g |x| |y|, g = (4 c + 6) u (c units a lane, u the
roundoff of the rows' arithmetic), scalars a few u of their terms; q0, q1, q2 and y~ follow from them and
a1..a4 by the product rule, constraint by constraint.  Sums over constraints and rows are
double-float or FP64.  The bound is tight enough to see one constraint: leaving one out of the
reference moves a coefficient by more than twice its bound (test on the CPU; for all constraints but
one in 200, whose dots are nearly 0), so that a dropped or doubled constraint fails the test.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from tests._util import mixed_instance

torch = pytest.importorskip("torch")
import paper_2407_15049_gb300 as L  # noqa: E402

RHO = 1.5
DT = {"fp64": (torch.float64, 2.0**-53), "fp32": (torch.float32, 2.0**-24), "bf16": (torch.bfloat16, 2.0**-24)}
SHAPES = [(7, 3), (33, 31), (65, 400), (257, 8)]
RANKS = [1, 8, 17, 24, 64, 128, 132]


def _reference(inst, R, D, y, u, skip=None):
    """a1..a4 in FP64 and their bounds; `skip`: a triplet left out."""
    C = sp.csr_matrix((inst.val, inst.colind, inst.rowptr), shape=(inst.n, inst.n))
    keep = np.ones(len(inst.row), bool)
    if skip is not None:
        keep[skip] = False
    i, j, con = inst.row[keep], inst.col[keep], inst.con[keep]
    fa = inst.aval[keep] * np.where(i == j, 1.0, 2.0)
    ni, nj = np.linalg.norm(R, axis=1), np.linalg.norm(D, axis=1)
    units = (R.shape[1] + 3) // 4
    g = (4 * ((units + 31) // 32) + 6) * u
    b, yk = inst.b[con], y[con]
    z = fa * np.sum(R[i] * R[j], axis=1) - b
    q1 = fa * np.sum(R[i] * D[j] + D[i] * R[j], axis=1)
    q2 = fa * np.sum(D[i] * D[j], axis=1)
    ez = np.abs(fa) * g * ni[i] * ni[j] + 4 * u * (np.abs(z) + np.abs(b))
    e1 = np.abs(fa) * g * (ni[i] * nj[j] + nj[i] * ni[j]) + 4 * u * np.abs(q1)
    e2 = np.abs(fa) * g * nj[i] * nj[j] + 4 * u * np.abs(q2)
    yt = yk - RHO * z
    ey = RHO * ez + 4 * u * (np.abs(yk) + RHO * np.abs(z))
    a1, a2, ay = np.abs(q1), np.abs(q2), np.abs(yt)
    CD, aCD = C @ D, abs(C) @ np.abs(D)
    gp = (int(np.diff(inst.rowptr).max(initial=0)) + 8 + 4 * ((units + 31) // 32)) * u
    a = np.array([0.5 * RHO * q2 @ q2, RHO * q1 @ q2, np.sum(CD * D) - yt @ q2 + 0.5 * RHO * q1 @ q1,
                  2 * np.sum(CD * R) - yt @ q1])
    bound = np.array([0.5 * RHO * np.sum(2 * a2 * e2 + e2**2), RHO * np.sum(a1 * e2 + a2 * e1 + e1 * e2),
                      gp * np.sum(aCD * np.abs(D)) + np.sum(ay * e2 + a2 * ey + ey * e2)
                      + 0.5 * RHO * np.sum(2 * a1 * e1 + e1**2),
                      2 * gp * np.sum(aCD * np.abs(R)) + np.sum(ay * e1 + a1 * ey + ey * e1)])
    return a, bound


def _inputs(n, r, dtype):
    f = lambda s: torch.as_tensor(np.random.default_rng(s).standard_normal((n, r))).to(dtype)  # noqa: E731
    return f(1), f(2)


@pytest.mark.parametrize("n,n_off", SHAPES)
@pytest.mark.parametrize("r", RANKS)
@pytest.mark.parametrize("prec", list(DT))
def test_bound_sees_each_constraint(n, n_off, r, prec):
    dtype, u = DT[prec]
    inst = mixed_instance(n, seed=n, n_off=n_off)
    R, D = (t.double().numpy() for t in _inputs(n, r, dtype))
    y = np.random.default_rng(3).standard_normal(inst.m)
    a, bound = _reference(inst, R, D, y, u)
    unseen = sum(np.all(np.abs(_reference(inst, R, D, y, u, skip=k)[0] - a) <= 2 * bound) for k in range(len(inst.row)))
    assert unseen <= len(inst.row) // 200


@pytest.mark.gpu
@pytest.mark.parametrize("n,n_off", SHAPES)
@pytest.mark.parametrize("r", RANKS)
@pytest.mark.parametrize("prec", list(DT))
def test_coefficients_within_the_bound(n, n_off, r, prec):
    dtype, u = DT[prec]
    inst = mixed_instance(n, seed=n, n_off=n_off)
    Rh, Dh = _inputs(n, r, dtype)
    pad = lambda t: torch.nn.functional.pad(t, (0, L.padded_ld(r) - r)).cuda().contiguous()  # noqa: E731
    y = np.random.default_rng(3).standard_normal(inst.m)
    want, bound = _reference(inst, Rh.double().numpy(), Dh.double().numpy(), y, u)
    ctx = L.lorads_create(inst)
    try:
        a, _ = L.lorads_linesearch_coeffs(ctx, pad(Rh), pad(Dh), torch.as_tensor(y, device="cuda"), RHO, r=r)
    finally:
        L.lorads_destroy(ctx)
    assert np.all(np.abs(a - want) <= bound + 1e-14 * np.abs(want)), (a - want, bound)
