"""amg_loss_grad's fused adjoint passes against the oracle's autograd, at the
sweep counts and level sizes where its buffers alias (no pre-smoothing, one
sweep, a coarsest level below and above 32 and 64 rows), and its repeats: the
second and later calls replay one captured graph and give the same bits, with
new coefficients, right-hand sides and cycle counts in between.  Bars: FP64
1e-10, FP32 1e-4 per V-cycle (the training path's bars)."""
import numpy as np
import pytest
import torch

import paper_2606_19251_gb300 as P
import workloads as W
from oracle import setup as OS
from oracle import solve as O
from oracle import train as OT
from tests.gpu_helpers import ctx_from_oracle

pytestmark = pytest.mark.gpu

C = np.array([0.62, 0.03, -0.01, -0.18, 0.02])
MESHES = {"grid_20_c16": (lambda: W.poisson5(20), 16), "fv_3k_c64": (lambda: W.fv_mesh("graded", 3000, 7)[0], 64),
          "cube_12_c200": (lambda: W.poisson7(12, 1e-1), 200)}


def _oracle(levels, c, f, nu1, nu2, n_vc):
    h = O.OHierarchy.of(levels)
    t = torch.tensor(c, requires_grad=True)
    L = OT.problem_loss(h, t, f, nu1, nu2, n_vc)
    L.backward()
    return float(L.detach()), t.grad.numpy()


@pytest.mark.parametrize("prec,tol", [(P.AMG_FP64, 1e-10), (P.AMG_FP32_IN_FP64, 1e-4)])
@pytest.mark.parametrize("nu1,nu2,n_vc", [(2, 2, 3), (0, 2, 2), (1, 0, 2), (3, 1, 1)])
@pytest.mark.parametrize("name", list(MESHES))
def test_adjoint_matches_autograd(name, nu1, nu2, n_vc, prec, tol):
    make, coarse = MESHES[name]
    levels = OS.build_hierarchy(make(), max_coarse=coarse)
    n = levels[0].A.n_rows
    ctx = ctx_from_oracle(levels, prec, nu1=nu1, nu2=nu2)
    try:
        rng = np.random.RandomState(3)
        first = {}
        for call in range(4):
            c = C * (1.0 + 0.05 * rng.standard_normal((len(levels), 5)) * (call % 2))
            f = W.rhs_zero_mean(call % 2, n)
            if call == 2:
                c = np.tile(C, (len(levels), 1))
            L, dc = P.amg_loss_grad(ctx, c, f, n_vc)
            Lr, dr = _oracle(levels, c, f, nu1, nu2, n_vc)
            assert abs(L - Lr) <= tol * n_vc * max(1.0, abs(Lr))
            assert np.abs(dc - dr).max() <= tol * n_vc * np.abs(dr).max()
            assert np.all(dc[-1] == 0.0)
            if call % 2 == 0:            # same inputs: the replay equals the first call's single launches
                assert first.setdefault("L", L) == L
                assert np.array_equal(first.setdefault("dc", dc), dc)
        L1, dc1 = P.amg_loss_grad(ctx, c, f, 1)       # another cycle count in between
        Lr, dr = _oracle(levels, c, f, nu1, nu2, 1)
        assert abs(L1 - Lr) <= tol * max(1.0, abs(Lr)) and np.abs(dc1 - dr).max() <= tol * np.abs(dr).max()
        L, dc2 = P.amg_loss_grad(ctx, c, f, n_vc)
        assert np.array_equal(dc, dc2)
    finally:
        P.amg_destroy(ctx)
