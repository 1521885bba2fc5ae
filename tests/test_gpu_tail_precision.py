"""The FP32 V-cycle's dense coarse tail loses nothing to the FP64 coarsest solve
that it replaces: held and summed in FP32 pairs, its result is the exact
V-cycle of the FP32 matrix values, rounded once.  Meshes whose tail starts on
level 0, right-hand sides in FP32: every entry within half an ulp of the FP64
reference on the same rounded values (2^-24 relative), plus 1e-10 of the
largest for the pairs' own rounding (48 bits, sums of up to 1024 terms)."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

import paper_2606_19251_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu

C = (0.75, 0.11, -0.004, -0.75, -0.42)


def _f32(x):
    return np.asarray(x, np.float32).astype(np.float64)


def _csr(d, ncol):
    return sp.csr_matrix((_f32(d["val"]), d["col"], d["row_ptr"]), shape=(d["n"], ncol))


def _reference(ctx, b, gnn):
    levels = [P.amg_get_level(ctx, l) for l in range(P.amg_num_levels(ctx))]

    def cycle(l, b):
        a, p = levels[l]
        if p is None:
            A = sp.csr_matrix((a["val"], a["col"], a["row_ptr"]), shape=(a["n"], a["n"])).toarray()
            return np.linalg.solve(A, b)
        A, Pm = _csr(a, a["n"]), _csr(p, p["nc"])
        if gnn:
            q = P.amg_get_smoother(ctx, l)
            M = sp.csr_matrix((_f32(q), a["col"], a["row_ptr"]), shape=A.shape)
        else:
            d = sp.csr_matrix((a["val"], a["col"], a["row_ptr"]), shape=A.shape).diagonal()
            M = sp.diags(_f32((2.0 / 3.0) / d))
        u = M @ b
        u = u + M @ (b - A @ u)
        u = u + Pm @ cycle(l + 1, Pm.T @ (b - A @ u))
        for _ in range(2):
            u = u + M @ (b - A @ u)
        return u

    return cycle(0, b)


@pytest.mark.parametrize("gnn", [False, True])
@pytest.mark.parametrize("n", [9, 16, 24])
def test_tail_is_exact_to_one_rounding(n, gnn):
    A = W.poisson5(n)
    ctx = P.amg_create(precision=P.AMG_FP32_IN_FP64)
    try:
        P.amg_setup(ctx, A)
        if gnn:
            P.amg_set_coeffs(ctx, np.tile(C, (P.amg_num_levels(ctx), 1)))
        b = _f32(W.rhs_uniform(n, A.n_rows))
        d_b, d_e = torch.tensor(b, device="cuda"), torch.empty(A.n_rows, dtype=torch.float64, device="cuda")
        P.amg_vcycle_device(ctx, d_b, d_e)
        e, want = d_e.cpu().numpy(), _reference(ctx, b, gnn)
        assert np.all(np.abs(e - want) <= 2.0 ** -24 * np.abs(want) + 1e-10 * np.abs(want).max())
    finally:
        P.amg_destroy(ctx)
