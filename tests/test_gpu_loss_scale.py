"""amg_loss_grad does not depend on the units of f and A: scaling either by a
power of two changes no bit of the loss or of dL/dc as long as the V-cycle's
own FP32 values stay normal numbers (they do up to 2^100 here).  The FP32
V-cycle's gradient sums run in FP32 pairs, whose low words leave the normal
range first."""
import numpy as np
import pytest

import paper_2606_19251_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [P.AMG_FP32_IN_FP64, P.AMG_FP64])
@pytest.mark.parametrize("mesh,coef", [(lambda: W.fv_mesh("graded", 6000, 3)[0], (0.70, 0.20, -0.08, -1.50, -0.70)),
                                       (lambda: W.poisson5(20), (0.75, 0.11, -0.004, -0.75, -0.42))],
                         ids=["graded_6k", "grid_20"])
def test_loss_and_gradient_are_scale_invariant(mesh, coef, prec):
    A = mesh()
    f = W.rhs_uniform(3, A.n_rows)

    def run(sa, sf):
        ctx = P.amg_create(precision=prec)
        try:
            P.amg_setup(ctx, W.CSR(A.n_rows, A.n_cols, A.row_ptr, A.col, A.val * sa))
            c = np.tile(coef, (P.amg_num_levels(ctx), 1))
            return P.amg_loss_grad(ctx, c, f * sf, 3)
        finally:
            P.amg_destroy(ctx)

    loss, dc = run(1.0, 1.0)
    for sa, sf in ((1.0, 2.0 ** -100), (1.0, 2.0 ** 100), (2.0 ** -100, 1.0), (2.0 ** 100, 1.0),
                   (2.0 ** 60, 2.0 ** -30)):
        ls, ds = run(sa, sf)
        assert ls == loss
        assert np.array_equal(ds, dc)
