"""What one poll of the device status costs: check_every iterations, whatever the captured graph holds.

A solve of one L-BFGS iteration enqueues two polls' work before it sees the first status, so the
kernels it enqueues are B + 2 (k I + g O): B for the start, I per iteration, O per outer step, k =
check_every and g graphs in a poll.
"""
import pytest
import torch

import paper_2407_15049_gb300 as L
import workloads as W

pytestmark = pytest.mark.gpu


def _launches(**params):
    n = 200
    inst = W.maxcut_instance(n, W.er_graph(n, 3 * n, 5, "pm1"))
    ctx = L.lorads_create(inst, L.default_params(tol=1e-300, **params))
    try:
        res = L.lorads_solve(ctx, W.initial_factor(inst, 8, 2), max_total_inner=1)
    finally:
        L.lorads_destroy(ctx)
    assert res["inner_iters"] == 1
    return res["kernel_launches"]


def test_polls_after_check_every_iterations():
    one, two, three, four = (_launches(check_every=k) for k in (1, 2, 3, 4))
    assert two - one == three - two == four - three > 0
    # five does not divide into graphs of up to four alike: five graphs of one iteration
    five, ten = _launches(check_every=5), _launches(check_every=10)
    assert five < ten
    outer = (five - one) // 8 - (two - one) // 2          # 5 I + 5 O - I - O, twice
    assert outer > 0 and five - one == 8 * ((two - one) // 2 + outer)


def test_a_graph_holds_no_more_iterations_than_an_inner_loop():
    step = _launches(check_every=2) - _launches(check_every=1)
    whole, single = _launches(check_every=4), _launches(check_every=4, max_inner=1)
    pair = _launches(check_every=4, max_inner=2)
    assert whole < pair < single
    assert single - whole == 3 * (pair - whole)             # 4, 2 and 1 graphs a poll
    assert step > 0
