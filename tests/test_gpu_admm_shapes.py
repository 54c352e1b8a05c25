"""The ADMM stage's constraint pass at the edges of its lane groups, through one CG step: the
step's residual holds w = y - rho (A(X V^T) - b), formed by groups that take their constraints
in batches of up to eight (rows of one unit a lane) or one at a time (wider rows).

X1 = X0 + (|r|^2 / <p, Q p>) r: the residual sums some tens of products of rows of up to 132
elements, and both sums of the step have terms of one sign, so the relative error of X1 is
below 1e3 units of roundoff of its largest term, 2e-13 in FP64 and 1e-4 in float; the bounds
are 1e-11 and 2e-4.
"""
import numpy as np
import pytest

from oracle import admm_oracle as A
from oracle import lorads_oracle as O
from tests._util import mixed_instance, rel_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2407_15049_gb300 as L  # noqa: E402


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("fp32", 2e-4)])
@pytest.mark.parametrize("n,n_off", [(7, 3), (33, 31), (65, 400), (257, 8)])
@pytest.mark.parametrize("r", [1, 5, 8, 17, 24, 33, 65, 128, 132])
def test_one_step_matches_oracle(n, n_off, r, prec, tol):
    dtype = torch.float64 if prec == "fp64" else torch.float32
    inst = mixed_instance(n, seed=n, n_off=n_off)
    P, ctx = O.Problem(inst), L.lorads_create(inst)
    rng = np.random.default_rng(r)
    rho = 2.5
    try:
        V, X = (torch.zeros((n, L.padded_ld(r)), dtype=dtype, device="cuda") for _ in range(2))
        for t in (V, X):
            t[:, :r] = torch.as_tensor(rng.standard_normal((n, r)) / np.sqrt(r), device="cuda").to(dtype)
        V0, X0 = (t[:, :r].double().cpu().numpy() for t in (V, X))
        y = rng.standard_normal(inst.m)
        want, _ = A.cg(P, V0, X0, A.system_rhs(P, V0, y, rho), rho, 1e-12, 1)
        steps = L.lorads_admm_cg(ctx, V, X, torch.as_tensor(y, device="cuda"), rho, cg_rel=1e-12, cg_max=1, r=r)
        assert steps == 1
        assert rel_err(X.double().cpu().numpy()[:, :r], want) <= tol
    finally:
        L.lorads_destroy(ctx)
