"""GPU parity of the V-cycle's dense coarse tail (csrc/tail.cuh) against the
FP64 oracle's level-by-level V-cycle.

Sizes sit at the edges of the rule and of the operator's layout: the tail
starting on level 0 with exactly 1024 rows, one level further down at 1025
rows and more, row counts around the 512-byte padding of B, no tail at all
(one level), uneven sweep counts.  Bars: FP64 1e-12 (the solve path's bar;
only the order of the sums differs), FP32 3e-5: about 50 rounded passes of
6e-8 each, with a factor 8 for the cancellation in b - A u.
"""
import numpy as np
import pytest
import torch

import paper_2606_19251_gb300 as P
import workloads as W
from oracle import setup as OS
from oracle import solve as O
from tests.gpu_helpers import ctx_from_oracle, oracle_hier, rel_err

pytestmark = pytest.mark.gpu

COEFFS = [0.62, 0.03, -0.01, -0.18, 0.02]
MESHES = {
    "grid_5": lambda: W.poisson5(5),                  # 25 rows: one level, no tail
    "grid_11": lambda: W.poisson5(11),                # 121 rows: tail on level 0, B narrower than one padded row
    "grid_32": lambda: W.poisson5(32),                # 1024 rows: the largest tail
    "box_1025": lambda: W.fv_mesh("graded", 1200, 3)[0],
    "cube_9": lambda: W.poisson7(9, 1e-2),            # 729 rows
    "band_6k": lambda: W.fv_mesh("band", 6000, 4, max_aspect=100.0)[0],
}


def _vcycle(ctx, b):
    d_b, d_e = torch.tensor(b, device="cuda"), torch.empty(len(b), dtype=torch.float64, device="cuda")
    P.amg_vcycle_device(ctx, d_b, d_e)
    torch.cuda.synchronize()
    return d_e.cpu().numpy()


def _oracle(levels, smoother, b, nu1, nu2):
    h = oracle_hier(levels, smoother, None if smoother == "jacobi" else np.tile(COEFFS, (len(levels), 1)))
    return O.vcycle(h, torch.from_numpy(b), torch.zeros(len(b), dtype=torch.float64), nu1, nu2).numpy()


@pytest.mark.parametrize("prec,tol", [(P.AMG_FP64, 1e-12), (P.AMG_FP32_IN_FP64, 3e-5)])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (0, 1), (3, 0)])
@pytest.mark.parametrize("name", list(MESHES))
def test_tail_vcycle_matches_oracle(name, nu1, nu2, prec, tol):
    A = MESHES[name]()
    levels = OS.build_hierarchy(A, max_coarse=40)
    ctx = ctx_from_oracle(levels, prec, nu1=nu1, nu2=nu2)
    try:
        b = W.rhs_uniform(5, A.n_rows)
        assert rel_err(_vcycle(ctx, b), _oracle(levels, "jacobi", b, nu1, nu2)) < tol
        P.amg_set_coeffs(ctx, np.tile(COEFFS, (len(levels), 1)))
        assert rel_err(_vcycle(ctx, b), _oracle(levels, "gnn", b, nu1, nu2)) < tol
        # new coefficients replace the operator; Jacobi's own stays
        P.amg_set_coeffs(ctx, np.tile([2.0 / 3.0, 0, 0, 0, 0], (len(levels), 1)))
        jac = _oracle(levels, "jacobi", b, nu1, nu2)
        assert rel_err(_vcycle(ctx, b), jac) < tol
        P.amg_set_jacobi(ctx)
        assert rel_err(_vcycle(ctx, b), jac) < tol
    finally:
        P.amg_destroy(ctx)


def test_captured_vcycle_follows_new_coefficients():
    A = MESHES["band_6k"]()
    levels = OS.build_hierarchy(A, max_coarse=40)
    ctx = ctx_from_oracle(levels, P.AMG_FP64)
    try:
        b = W.rhs_uniform(6, A.n_rows)
        d_b, d_e = torch.tensor(b, device="cuda"), torch.zeros(A.n_rows, dtype=torch.float64, device="cuda")
        P.amg_set_coeffs(ctx, np.tile([2.0 / 3.0, 0, 0, 0, 0], (len(levels), 1)))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            P.amg_vcycle_device(ctx, d_b, d_e)
        P.amg_loss_grad(ctx, np.tile(COEFFS, (len(levels), 1)), b, 1)      # leaves the tail's operator behind
        # loss_grad assembles Q^-1 and M A as amg_set_coeffs does: the replay runs the new smoother
        g.replay()
        torch.cuda.synchronize()
        want = _oracle(levels, "gnn", b, 2, 2)
        assert rel_err(d_e.cpu().numpy(), want) < 1e-12
        assert rel_err(_vcycle(ctx, b), want) < 1e-12
    finally:
        P.amg_destroy(ctx)
