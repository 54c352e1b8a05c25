"""The root of the exact line search over coefficients of many magnitudes: searches that end
after a few Newton steps and searches that go through long runs of bisections, which a warp
takes several at a time.

The search ends where f' is zero as evaluated or where the bracket is 4 units of roundoff
wide, so |f'(tau)|, in exact arithmetic, is at most a few units of roundoff of its terms'
magnitudes plus 4 of |tau f''(tau)|: 8 units of both.  Of the positive roots it takes the one
of the lowest quartic value: no higher than the oracle's, to 1e-9 of the terms' magnitudes.
"""
from fractions import Fraction

import numpy as np
import pytest

import workloads as W
from oracle import lorads_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_2407_15049_gb300 as L  # noqa: E402

EPS = 2.0 ** -52


def _rows(values):
    t = torch.zeros((values.shape[0], L.padded_ld(values.shape[1])), dtype=torch.float64, device="cuda")
    t[:, :values.shape[1]] = torch.as_tensor(values, device="cuda")
    return t


@pytest.mark.parametrize("scale_d", [1e-4, 1e-2, 1.0, 1e2, 1e5])
@pytest.mark.parametrize("scale_y", [0.0, 1.0, 1e3])
@pytest.mark.parametrize("rho", [0.3, 40.0])
def test_root_is_a_root_and_the_lowest(scale_d, scale_y, rho):
    inst = W.maxcut_instance(5, (np.array([0, 0, 1, 2, 3]), np.array([1, 2, 3, 4, 4]), np.array([1.0, -2.0, 0.5, 1.0, 3.0])))
    ctx = L.lorads_create(inst)
    rng = np.random.default_rng(int(scale_y) + int(10 * rho))
    found = 0
    try:
        for _ in range(24):
            R, D = rng.standard_normal((5, 3)), scale_d * rng.standard_normal((5, 3))
            y = torch.as_tensor(scale_y * rng.standard_normal(inst.m), device="cuda")
            a, tau = L.lorads_linesearch_coeffs(ctx, _rows(R), _rows(D), y, rho, r=3)
            want = O.quartic_step(a)
            assert (tau > 0.0) == (want > 0.0)
            if tau == 0.0:
                continue
            found += 1
            t, (a1, a2, a3, a4) = Fraction(float(tau)), (Fraction(float(v)) for v in a)
            terms = [4 * a1 * t**3, 3 * a2 * t**2, 2 * a3 * t, a4]
            curve = abs(12 * a1 * t**2 + 6 * a2 * t + 2 * a3) * t
            assert abs(sum(terms)) <= 8 * EPS * (sum(abs(v) for v in terms) + curve)
            mags = float(sum(abs(v) for v in terms) * t)
            assert O.quartic_value(a, tau) <= O.quartic_value(a, want) + 1e-9 * mags
        assert found > 4
    finally:
        L.lorads_destroy(ctx)
