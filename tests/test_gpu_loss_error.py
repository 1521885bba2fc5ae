"""amg_loss_grad sets its coefficients without a wait; when a later step of the
call fails, the assembly has still ended before the call returns, so that the
next call, on whatever stream, finds it complete.  The failure is an error code
of cudaMalloc from a preloaded shim (a child process); nothing runs out of
memory."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

SHIM = r"""
#include <dlfcn.h>
#include <stddef.h>
static int armed = 0, failed = 0, waits = 0;
/* the runtime that the library has loaded (it is not in the global scope) */
static void *real_of(const char *name) { return dlsym(dlopen("libcudart.so.13", RTLD_LAZY), name); }
void shim_arm(void) { armed = 1; failed = waits = 0; }
int shim_failed(void) { return failed; }
int shim_waits(void) { return waits; }
int cudaMalloc(void **p, size_t n) {
    static int (*real)(void **, size_t);
    if (armed) { armed = 0; failed = 1; return 2; }   /* cudaErrorMemoryAllocation */
    if (!real) real = (int (*)(void **, size_t))real_of("cudaMalloc");
    return real(p, n);
}
int cudaStreamSynchronize(void *s) {
    static int (*real)(void *);
    if (!real) real = (int (*)(void *))real_of("cudaStreamSynchronize");
    if (failed) ++waits;
    return real(s);
}
"""

CHILD = """
import ctypes, os
import numpy as np
import paper_2606_19251_gb300 as P
import workloads as W
shim = ctypes.CDLL(os.environ["LD_PRELOAD"])
A = W.poisson5(40)
b = W.rhs_uniform(1, A.n_rows)
ctx, ref = P.amg_create(), P.amg_create()
for c in (ctx, ref):
    P.amg_setup(c, A)
nl = P.amg_num_levels(ctx)
new = np.tile([0.70, 0.01, 0.0, -0.10, 0.01], (nl, 1))
P.amg_set_coeffs(ctx, np.tile([0.62, 0.03, -0.01, -0.18, 0.02], (nl, 1)))
shim.shim_arm()
try:
    P.amg_loss_grad(ctx, new, b, 2)
    raise SystemExit("no error")
except P.AmgError as e:
    assert e.code == P.AMG_ERR_CUDA, e
assert shim.shim_failed() == 1
assert shim.shim_waits() >= 1, "returned while the assembly may still run"
P.amg_set_coeffs(ref, new)          # the coefficients of the failed call are in force
(s0, x0, h0), (s1, x1, h1) = P.amg_solve(ctx, b), P.amg_solve(ref, b)
assert s0 == s1 == P.AMG_OK and np.array_equal(x0, x1) and np.array_equal(h0, h1)
print("child ok", P.amg_loss_grad(ctx, new, b, 2)[0])
"""


def test_failed_allocation_leaves_a_complete_assembly(tmp_path):
    src, so = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout + r.stderr
