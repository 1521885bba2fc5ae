"""The residual history holds every entry that a call may write: a solve writes
max_iter + 1, the probe solves of amg_judge and amg_reroute n_cycles + 1 (up to
10001) whatever the context's max_iter."""
import os
import subprocess

import numpy as np
import pytest

import paper_2606_19251_gb300 as P
import workloads as W
from paper_2606_19251_gb300 import _build

SOURCE = """
#include "ctx.cuh"
static_assert(amg::kMaxProbeCycles == 10000, "the header's limit of n_cycles");
static_assert(amg::hist_capacity(0) == 10001 && amg::hist_capacity(500) == 10001, "probe solves");
static_assert(amg::hist_capacity(10000) == 10001 && amg::hist_capacity(10001) == 10002, "the longer of both");
static_assert(amg::hist_capacity(100000) == 100001, "solves");
"""


def test_capacity_covers_solves_and_probes(tmp_path):
    src = tmp_path / "capacity.cu"
    src.write_text(SOURCE)
    r = subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-c", str(src), "-o", str(tmp_path / "capacity.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    with open(os.path.join(_build.CSRC, "amg_solver.cu")) as f:
        text = f.read()
    # the history is laid out with that capacity, and both probes refuse more
    assert "hist_cap = hist_capacity(c->opt.max_iter)" in text
    assert text.count("n_cycles > kMaxProbeCycles") == 2


@pytest.mark.gpu
@pytest.mark.parametrize("max_iter", [0, 5])
def test_probes_longer_than_max_iter(max_iter):
    """A context with a short max_iter judges as one that allows the cycles."""
    A = W.poisson5(24)
    b = W.rhs_uniform(3, A.n_rows)
    out = []
    for mi in (max_iter, 700):
        ctx = P.amg_create(max_iter=mi)
        try:
            P.amg_setup(ctx, A)
            P.amg_set_coeffs(ctx, np.tile([0.62, 0.03, -0.01, -0.18, 0.02], (P.amg_num_levels(ctx), 1)))
            out.append((P.amg_judge(ctx, b, 12), P.amg_judge(ctx, b, 600), P.amg_reroute(ctx, b, 650)))
        finally:
            P.amg_destroy(ctx)
    assert out[0] == out[1]


@pytest.mark.parametrize("call,kw", [("amg_solve", dict(max_iter=3)), ("amg_solve_device", dict(hist_cap=4)),
                                     ("amg_solve", {}), ("amg_solve_device", {})])
def test_binding_gives_room_for_any_history(monkeypatch, call, kw):
    """The library writes one entry per cycle of the context's max_iter (at most
    100000), whatever the caller expects: the buffer it gets holds them all."""
    from paper_2606_19251_gb300 import api
    sizes = []

    class Lib:
        def __getattr__(self, name):
            return lambda *a: 0

    monkeypatch.setattr(api, "lib", lambda: Lib())
    monkeypatch.setattr(api, "_dev", lambda t: None)
    monkeypatch.setattr(api, "_stream", lambda s: None)
    monkeypatch.setattr(api, "_dptr", lambda a: sizes.append(a.size))
    b = np.zeros(7)
    api.amg_solve(None, b, **kw) if call == "amg_solve" else api.amg_solve_device(None, b, b, **kw)
    assert max(sizes) == 100001
