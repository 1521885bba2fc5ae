"""The V-cycle's dense coarse tail at the edges of its rule and of its layout,
and when it is formed.

Row counts are exact (leading blocks of a mesh): next to the 512-byte padding
of B's rows (63/64/65 in FP64, 127/128/129 in FP32) and to the largest level
(1023/1024/1025).  Kernel launches tell where the tail starts: on level 0 a
V-cycle is the operator alone (and two conversions in FP32).  Bars: FP64 1e-12,
FP32 3e-5 (the V-cycle's)."""
import numpy as np
import pytest
import torch

import paper_2606_19251_gb300 as P
import workloads as W
from oracle import setup as OS
from oracle import solve as O
from tests.gpu_helpers import ctx_from_oracle, oracle_hier, rel_err
from tests.test_gpu_train_tiles import _leading

pytestmark = pytest.mark.gpu

PREC = [(P.AMG_FP64, 1e-12), (P.AMG_FP32_IN_FP64, 3e-5)]
COEFFS = [0.62, 0.03, -0.01, -0.18, 0.02]
ROWS, WORK = 1024, {P.AMG_FP64: 1.5e6, P.AMG_FP32_IN_FP64: 4e6}


def _tail_level(levels, work):
    """The rule: the finest level from which on all levels fit."""
    nL, best = levels[-1].A.n_rows, -1
    rows, entries = nL, int(levels[-1].A.row_ptr[-1])
    for l in range(len(levels) - 2, -1, -1):
        n = levels[l].A.n_rows
        rows, entries = rows + n, entries + int(levels[l].A.row_ptr[-1])
        if n > ROWS or 96 * rows > 220 * 1024 or n * nL * nL > 2 ** 27 or n * entries > work:
            break
        best = l
    return best


def _v(ctx, b):
    d_b, d_e = torch.tensor(b, device="cuda"), torch.empty(len(b), dtype=torch.float64, device="cuda")
    before = P.amg_launch_count()
    P.amg_vcycle_device(ctx, d_b, d_e)
    torch.cuda.synchronize()
    return d_e.cpu().numpy(), P.amg_launch_count() - before


def _oracle(levels, b, setter):
    h = O.OHierarchy.of(levels)
    setter(h)
    return O.vcycle(h, torch.from_numpy(b), torch.zeros(len(b), dtype=torch.float64), 2, 2).numpy()


def _check(ctx, levels, b, setter, prec, tol, tail):
    want = _oracle(levels, b, setter)
    e, first = _v(ctx, b)                        # forms B
    assert rel_err(e, want) < tol
    e2, n = _v(ctx, b)
    assert np.array_equal(e, e2)
    whole = 1 if prec == P.AMG_FP64 else 3
    assert (n == whole) if tail == 0 else (n > whole)
    return first - n                             # kernels that formed B


@pytest.mark.parametrize("prec,tol", PREC)
@pytest.mark.parametrize("rows", [63, 64, 65, 127, 128, 129, 1023, 1024, 1025])
def test_row_counts_at_the_edges(rows, prec, tol):
    A = _leading(W.poisson5(40), rows)
    assert A.n_rows == rows
    levels = OS.build_hierarchy(A, max_coarse=40)
    ctx = ctx_from_oracle(levels, prec)
    try:
        b = W.rhs_uniform(rows, rows)
        assert _check(ctx, levels, b, lambda h: h.set_jacobi(), prec, tol, _tail_level(levels, np.inf)) == 0
        small = _tail_level(levels, WORK[prec])
        P.amg_set_coeffs(ctx, np.tile(COEFFS, (len(levels), 1)))
        formed = _check(ctx, levels, b, lambda h: h.set_pseudo_inverse(np.tile(COEFFS, (len(levels), 1))), prec, tol, small)
        assert formed == (1 if small >= 0 else 0)
        P.amg_set_jacobi(ctx, 0.55)              # a changed omega: B again, within the work for new values
        formed = _check(ctx, levels, b, lambda h: h.set_jacobi(0.55), prec, tol, small)
        assert formed == (1 if small >= 0 else 0)
    finally:
        P.amg_destroy(ctx)


@pytest.mark.parametrize("prec,tol", PREC)
@pytest.mark.parametrize("rows,max_coarse,tail", [(600, 310, 0), (1000, 510, -1)])
def test_large_coarsest_level(rows, max_coarse, tail, prec, tol):
    """Coarsest levels of some hundred rows: below and above the bound of their solves."""
    levels = OS.build_hierarchy(_leading(W.poisson5(40), rows), max_coarse=max_coarse)
    assert len(levels) == 2 and levels[-1].A.n_rows > 250 and _tail_level(levels, np.inf) == tail
    ctx = ctx_from_oracle(levels, prec, max_coarse=max_coarse)
    try:
        b = W.rhs_uniform(2, rows)
        _check(ctx, levels, b, lambda h: h.set_jacobi(), prec, tol, tail)
    finally:
        P.amg_destroy(ctx)


def test_fp64_tail_on_a_finest_level_past_l2():
    """The bound on the finest level is one of FP32 rounding: an FP64 V-cycle has its tail there too."""
    ctx = P.amg_create(precision=P.AMG_FP64)
    try:
        A = W.poisson5(1040)
        P.amg_setup_device(ctx, A, 0, P.AMG_SPLIT_RS_BLOCKS)
        P.amg_set_coeffs(ctx, np.tile(COEFFS, (P.amg_num_levels(ctx), 1)))
        b = W.rhs_uniform(1, A.n_rows)
        (e, first), (e2, n) = _v(ctx, b), _v(ctx, b)
        assert first == n + 1 and np.array_equal(e, e2)
    finally:
        P.amg_destroy(ctx)


def test_calls_that_set_values_form_no_operator():
    """amg_set_coeffs and amg_set_jacobi launch the assembly alone."""
    levels = OS.build_hierarchy(W.fv_mesh("graded", 3000, 3)[0], max_coarse=40)
    ctx = ctx_from_oracle(levels, P.AMG_FP32_IN_FP64)
    try:
        for call, kernels in ((lambda: P.amg_set_coeffs(ctx, np.tile(COEFFS, (len(levels), 1))), 2),
                              (lambda: P.amg_set_jacobi(ctx, 0.6), len(levels))):
            before = P.amg_launch_count()
            call()
            assert P.amg_launch_count() - before == kernels
    finally:
        P.amg_destroy(ctx)


@pytest.mark.parametrize("prec,tol", PREC)
def test_operator_follows_predictions_and_omega(prec, tol):
    """Predictions only mark B as stale; V-cycles and solves after them, and
    after a change of omega, use the new values."""
    A = W.fv_mesh("graded", 4000, 5)[0]
    ctx, ref = P.amg_create(precision=prec), P.amg_create(precision=prec)
    try:
        for c in (ctx, ref):
            P.amg_setup(c, A)
        b = W.rhs_uniform(4, A.n_rows)
        last = None
        for seed in (1, 2, 1):
            P.gnn_load_params(ctx, W.gcin_init_params(seed).astype(np.float32))
            P.amg_set_coeffs(ref, P.gnn_predict_coeffs(ctx))
            for _ in range(3):
                e = _v(ctx, b)[0]
                assert rel_err(e, _v(ref, b)[0]) < tol
            assert last is None or rel_err(e, last) > 1e-4
            last = e
        for omega in (0.5, 2.0 / 3.0, 0.6):
            for c in (ctx, ref):
                P.amg_set_jacobi(c, omega)
            (s0, x0, h0), (s1, x1, h1) = P.amg_solve(ctx, b), P.amg_solve(ref, b)
            assert s0 == s1 == P.AMG_OK and np.array_equal(x0, x1) and np.array_equal(h0, h1)
            h = OS.build_hierarchy(A)
            assert rel_err(_v(ctx, b)[0], _oracle(h, b, lambda o: o.set_jacobi(omega))) < tol
    finally:
        P.amg_destroy(ctx)
        P.amg_destroy(ref)
