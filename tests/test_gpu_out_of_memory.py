"""A solve whose state does not fit returns an error, again when it is repeated, and leaves the context usable."""
import pytest
import torch

import paper_2407_15049_gb300 as L
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [L.LORADS_FP64, L.LORADS_MIXED])
def test_a_state_that_does_not_fit(prec):
    n, wide = 200000, 512            # the state takes 7 GB (mixed) to 11 GB (FP64) at 512 columns
    inst = W.maxcut_instance(n, W.er_graph(n, n, 1, "pm1"))
    ctx = L.lorads_create(inst, L.default_params(prec=prec))
    try:
        torch.cuda.empty_cache()
        held = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
        for _ in range(2):
            with pytest.raises(L.LoradsError, match="cudaMalloc"):
                L.lorads_solve(ctx, None, r0=wide, max_total_inner=1)
        with pytest.raises(L.LoradsError):
            L.lorads_get_solution(ctx, inst.n, inst.m)
        del held
        torch.cuda.empty_cache()
        res = L.lorads_solve(ctx, None, r0=8, max_total_inner=3)
        R, _ = L.lorads_get_solution(ctx, inst.n, inst.m)
    finally:
        L.lorads_destroy(ctx)
    assert res["inner_iters"] == 3 and R.shape == (n, 8)
