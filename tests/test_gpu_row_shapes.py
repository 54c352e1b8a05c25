"""The constraint pass and the gradient product at the edges of their lane groups: row
widths of one lane to several units a lane, constraint and row counts around the batch of
eight and the warp, degrees around the entries in flight.

Tolerances: normwise 1e-12 in FP64 and 1e-5 in FP32 and BF16 against the FP64 oracle on the
same rounded inputs (a dot of r <= 132 products and a sum of some tens of rows have a
rounding error below 1e3 units of roundoff: 2e-13 and 6e-5 at worst, 1e-14 and 1e-6 as it
grows in practice), the bounds of the other kernel tests.
"""
import numpy as np
import pytest

from oracle import lorads_oracle as O
from tests._util import mixed_instance, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2407_15049_gb300 as L  # noqa: E402

DT = {"fp64": (torch.float64, 1e-12), "fp32": (torch.float32, 1e-5), "bf16": (torch.bfloat16, 1e-5)}
RANKS = [1, 5, 8, 16, 17, 24, 33, 64, 65, 128, 132]


def _factor(n, r, seed, dtype):
    t = torch.zeros((n, L.padded_ld(r)), dtype=dtype, device="cuda")
    t[:, :r] = torch.as_tensor(np.random.default_rng(seed).standard_normal((n, r)), device="cuda").to(dtype)
    return t, t[:, :r].double().cpu().numpy()


@pytest.mark.parametrize("prec", list(DT))
@pytest.mark.parametrize("n,n_off", [(7, 3), (33, 31), (65, 400), (257, 8)])
@pytest.mark.parametrize("r", RANKS)
def test_row_shapes(n, n_off, r, prec):
    dtype, tol = DT[prec]
    inst = mixed_instance(n, seed=n, n_off=n_off)
    P, ctx = O.Problem(inst), L.lorads_create(inst)
    try:
        U, Ur = _factor(n, r, 1, dtype)
        V, Vr = _factor(n, r, 2, dtype)
        y = np.random.default_rng(3).standard_normal(inst.m)
        yd = torch.as_tensor(y, device="cuda")
        for A, Ar, B, Br in ((U, Ur, V, Vr), (U, Ur, U, Ur)):
            out = torch.full((inst.m,), float("nan"), dtype=torch.float64, device="cuda")
            L.lorads_constraint_eval(ctx, A, B, out, r=r)
            assert rel_err(out.cpu().numpy(), O.constraint_map(P, Ar, Br)) <= tol
        for v, vd in ((None, None), (y, yd)):
            out = torch.full((n, U.shape[1]), float("nan"), dtype=torch.float64 if prec == "fp64" else torch.float32,
                             device="cuda")
            L.lorads_spmm(ctx, U, vd, out, r=r)
            got = out.double().cpu().numpy()
            assert rel_err(got[:, :r], O.spmm(P, Ur, v)) <= tol and np.all(got[:, r:] == 0.0)
        a, _ = L.lorads_linesearch_coeffs(ctx, U, V, yd, 1.5, r=r)
        want, parts = O.linesearch_coeffs(P, Ur, Vr, y, 1.5)
        q0, q1, q2 = (np.abs(parts[k]) for k in ("q0", "q1", "q2"))
        w = np.abs(y) + 1.5 * q0
        C = abs(P.C)
        scale = np.array([0.75 * q2 @ q2, 1.5 * q1 @ q2,
                          np.sum((C @ np.abs(Vr)) * np.abs(Vr)) + w @ q2 + 0.75 * q1 @ q1,
                          2 * np.sum((C @ np.abs(Vr)) * np.abs(Ur)) + w @ q1])
        # the products of a constraint carry the error of its dots, not of their sums
        dots = np.sqrt(np.sum(Ur**2) * np.sum(Vr**2)) + np.sum(Vr**2)
        assert np.all(np.abs(a - want) <= tol * (scale + dots * (1 + np.linalg.norm(w) + dots)))
    finally:
        L.lorads_destroy(ctx)
