"""amg_vcycle_device over many calls: single launches at first, then one captured
graph.  The change is invisible: the same bits before and after it, with new
coefficients, a changed omega (whose tail may start on another level) and
another smoother in between."""
import numpy as np
import pytest
import torch

import paper_2606_19251_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu

C1, C2 = [0.62, 0.03, -0.01, -0.18, 0.02], [0.70, 0.01, 0.0, -0.10, 0.01]


@pytest.mark.parametrize("prec", [P.AMG_FP64, P.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("n", [30, 100])
def test_calls_before_and_after_the_capture_agree(n, prec):
    A = W.poisson5(n)
    b = torch.tensor(W.rhs_uniform(1, A.n_rows), device="cuda")
    e = torch.empty_like(b)

    def v(ctx):
        P.amg_vcycle_device(ctx, b, e)
        torch.cuda.synchronize()
        return e.cpu().numpy()

    ctx = P.amg_create(precision=prec)
    try:
        P.amg_setup(ctx, A)
        nl = P.amg_num_levels(ctx)
        for setter in (lambda c: P.amg_set_jacobi(c), lambda c: P.amg_set_coeffs(c, np.tile(C1, (nl, 1))),
                       lambda c: P.amg_set_coeffs(c, np.tile(C2, (nl, 1))), lambda c: P.amg_set_chebyshev(c, 2),
                       lambda c: P.amg_set_jacobi(c, 0.5), lambda c: P.amg_set_jacobi(c, 0.6)):
            setter(ctx)
            fresh = P.amg_create(precision=prec)
            try:
                P.amg_setup(fresh, A)
                setter(fresh)
                want = v(fresh)
            finally:
                P.amg_destroy(fresh)
            for _ in range(15):
                assert np.array_equal(v(ctx), want)
    finally:
        P.amg_destroy(ctx)
