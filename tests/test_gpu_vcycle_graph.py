"""amg_vcycle_device repeats: the second and later calls replay one captured
graph.  They give the same bits as the first call's single launches, follow
changes of coefficients, smoother, Chebyshev degree and hierarchy, and run on
another stream and inside a caller's own capture."""
import numpy as np
import pytest
import torch

import paper_2606_19251_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu

C1 = [0.62, 0.03, -0.01, -0.18, 0.02]
C2 = [0.70, 0.01, 0.0, -0.10, 0.01]


def _v(ctx, b):
    d_e = torch.empty_like(b)
    P.amg_vcycle_device(ctx, b, d_e)
    torch.cuda.synchronize()
    return d_e.cpu().numpy()


def _first(A, prec, setter, b):
    """The first call of a fresh context: single launches."""
    ctx = P.amg_create(precision=prec)
    try:
        P.amg_setup(ctx, A)
        setter(ctx)
        return _v(ctx, b)
    finally:
        P.amg_destroy(ctx)


@pytest.mark.parametrize("prec", [P.AMG_FP64, P.AMG_FP32_IN_FP64])
@pytest.mark.parametrize("n", [12, 70])
def test_repeats_equal_the_first_call(n, prec):
    A = W.poisson5(n)
    b = torch.tensor(W.rhs_uniform(1, A.n_rows), device="cuda")
    b2 = torch.tensor(W.rhs_uniform(2, A.n_rows), device="cuda")
    ctx = P.amg_create(precision=prec)
    try:
        P.amg_setup(ctx, A)
        nl = P.amg_num_levels(ctx)
        setters = [lambda c: P.amg_set_jacobi(c), lambda c: P.amg_set_coeffs(c, np.tile(C1, (nl, 1))),
                   lambda c: P.amg_set_chebyshev(c, 2), lambda c: P.amg_set_chebyshev(c, 3),
                   lambda c: P.amg_set_coeffs(c, np.tile(C2, (nl, 1))), lambda c: P.amg_set_jacobi(c, 0.5)]
        for s in setters:
            s(ctx)
            want, want2 = _first(A, prec, s, b), _first(A, prec, s, b2)
            for _ in range(3):
                assert np.array_equal(_v(ctx, b), want)
                assert np.array_equal(_v(ctx, b2), want2)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            e = torch.empty_like(b)
            P.amg_vcycle_device(ctx, b, e)
        side.synchronize()
        assert np.array_equal(e.cpu().numpy(), _first(A, prec, setters[-1], b))
        A2 = W.poisson5(n + 1)                       # another hierarchy in the same context
        P.amg_setup(ctx, A2)
        b3 = torch.tensor(W.rhs_uniform(3, A2.n_rows), device="cuda")
        want = _first(A2, prec, lambda c: None, b3)
        for _ in range(3):
            assert np.array_equal(_v(ctx, b3), want)
    finally:
        P.amg_destroy(ctx)
