"""Performance cases: the calls a pressure-solver user of this library makes.

A case is one public call (or the short fixed sequence a program repeats) on a
seeded mesh: a whole solve, one prediction of the smoother's coefficients, a
prediction with the solve that follows it, one V-cycle as a preconditioner, or
one training evaluation.  Meshes are

* "tri":   vertex-centred finite volumes on a graded (10:1) triangulation with
           jittered vertices and, with `aspect` > 1, a band of stretched cells;
           couplings are the cotangent two-point fluxes, Dirichlet on x = 1 and
           Neumann elsewhere.  About 7 entries per row, 4 to 9.  Unknowns are
           numbered column by column (the locality order large meshes come in);
* "fv":    the benchmark's graded Delaunay mesh (workloads.fv_mesh);
* "grid2": 5-point grid with a disk of low conductivity, Dirichlet all round;
* "grid3": 7-point grid with a sphere of low conductivity, Dirichlet all round.

Contexts, hierarchies, network parameters and right-hand sides are prepared
once, as a program with a fixed mesh keeps them; coefficients of the
pseudo-inverse smoother are given rows where the case is not about predicting
them.  FP32 results (the mixed-precision V-cycle, the network's coefficients)
are handed on as the float32 they were computed in.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2606_19251_gb300 as P
import workloads as W
from paper_2606_19251_gb300 import autograd as AG

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WEIGHTS = os.path.join(ROOT, "paper_2606_19251_gb300", "weights")
OMEGA = 2.0 / 3.0
# coefficient row (d0, d1, d2, o1, o2) of the pseudo-inverse smoother on every
# level where a case takes it as given: of the form the committed networks
# predict for these meshes, and fewer V-cycles than Jacobi on all of them
COEFFS = {"tri": (0.70, 0.20, -0.08, -1.50, -0.70), "grid2": (0.75, 0.11, -0.004, -0.75, -0.42),
          "grid3": (0.75, 0.11, -0.004, -0.75, -0.42)}


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the smallest system: 64 x 64 grid, all FP64; latency of a whole solve
        dict(name="solve_grid64_fp64", op="solve", mesh="grid2", n=4096, precision="fp64", smoother="jacobi",
             outer="refine", setup="host"),
        # the 50k-point graded mesh of the benchmark: predict the smoother, then solve with it
        dict(name="step_fv50k", op="step", mesh="fv", n=50000, precision="mixed", smoother="gnn", outer="refine",
             setup="host", hidden=64, net="bf16"),
        # 3D grid, conjugate gradients around the V-cycle, levels built on the GPU
        dict(name="solve_grid3_262k_cg", op="solve", mesh="grid3", n=262144, precision="mixed", smoother="jacobi",
             outer="pcg", setup="device"),
        # the 2.5M-point mesh with cells stretched 1000:1: the HBM-sized solve with the learned smoother's form
        dict(name="solve_band2500k_gnn", op="solve", mesh="tri", n=2500000, aspect=1000, precision="mixed",
             smoother="gnn", outer="refine", setup="device"),
        # one V-cycle as the preconditioner of a caller's own Krylov loop: small, ordinary, large
        dict(name="vcycle_tri9k_gnn", op="vcycle", mesh="tri", n=9001, precision="mixed", smoother="gnn",
             setup="host"),
        dict(name="vcycle_tri280k_gnn", op="vcycle", mesh="tri", n=280000, aspect=100, precision="mixed",
             smoother="gnn", setup="device"),
        dict(name="vcycle_grid1m_jacobi", op="vcycle", mesh="grid2", n=1050625, precision="mixed", smoother="jacobi",
             setup="device"),
        # coefficient prediction alone: new matrix values on a known mesh, default network and precision
        dict(name="predict_tri50k", op="predict", mesh="tri", n=50000, setup="host", hidden=64, net="bf16"),
        dict(name="predict_tri1200k", op="predict", mesh="tri", n=1200000, aspect=100, setup="device", hidden=64,
             net="bf16"),
        # the halved network of the structured meshes, FP32 linears
        dict(name="predict_grid3_110k_h32", op="predict", mesh="grid3", n=110592, setup="device", hidden=32,
             net="fp32"),
        # training: loss and coefficient gradient of one mesh through three V-cycles
        dict(name="loss_tri12k", op="loss", mesh="tri", n=12000, precision="mixed", setup="host", n_vc=3),
        # training: network forward, per-mesh losses, backward to the parameters, mini-batch of five meshes
        dict(name="train_batch5", op="train", mesh="tri", n=8000, precision="mixed", setup="host", n_vc=3, batch=5,
             hidden=64, net="fp32"),
    ]


def draw(rng):
    """One more case of the same ranges (sizes over their logarithm)."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["solve", "solve", "step", "vcycle", "vcycle", "vcycle", "predict", "predict", "loss", "train"])
    mesh = rng.choice(["tri", "tri", "grid2", "grid3"])
    c = dict(op=op, mesh=mesh)
    if mesh == "tri":
        c["aspect"] = rng.choice([1, 1, 100, 1000])
    if op in ("loss", "train"):
        c.update(n=size(2000, 20000), precision="mixed", setup="host", n_vc=rng.choice([1, 3]))
        if op == "train":
            c.update(batch=rng.randint(2, 6), hidden=rng.choice([64, 32]), net=rng.choice(["fp32", "fp32", "bf16"]))
        return c
    if op == "predict":
        c.update(n=size(4000, 1200000), hidden=rng.choice([64, 64, 32]), net=rng.choice(["bf16", "bf16", "fp32"]))
    elif op == "step":
        c = dict(op=op, mesh="fv", n=size(8000, 100000), precision="mixed", smoother="gnn", outer="refine",
                 hidden=64, net="bf16")
    else:
        c.update(n=size(4000, 1500000), precision=rng.choice(["mixed", "mixed", "mixed", "fp64"]),
                 smoother=rng.choice(["jacobi", "gnn"]))
        if op == "solve":
            c["outer"] = rng.choice(["refine", "pcg"])
    c["setup"] = "host" if c["n"] <= 60000 or op == "step" else "device"
    return c


# ----------------------------------------------------------------------------
# meshes (on the GPU, from the seed alone)
# ----------------------------------------------------------------------------
class _Matrix:
    def __init__(self, row_ptr, col, val):
        self.n_rows = self.n_cols = int(row_ptr.numel()) - 1
        self.row_ptr, self.col, self.val = (row_ptr.cpu().numpy().astype(np.int32), col.cpu().numpy().astype(np.int32),
                                            val.cpu().numpy())


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _slots_to_csr(cols, vals, keep):
    """CSR from per-row slots (n, k) in ascending column order."""
    n = cols.shape[0]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=cols.device)
    row_ptr[1:] = torch.cumsum(keep.sum(1), 0)
    return _Matrix(row_ptr, cols[keep], vals[keep])


def _tri(n, aspect, seed):
    ny = max(8, int(round(math.sqrt(n))))
    nx = max(8, int(round(n / ny)))
    dev, f64 = "cuda", torch.float64
    g = _gen(seed)
    h = 1.0 / nx
    j = torch.arange(ny - 1, dtype=f64, device=dev)
    dy = torch.full((ny - 1,), h, dtype=f64, device=dev)
    if aspect > 1:
        dy = torch.clamp(h / aspect * 1.1 ** (j - (ny - 1) // 2).abs(), max=h)
    ly = torch.cat([dy[:1], torch.minimum(dy[1:], dy[:-1]), dy[-1:]])          # spacing at each vertex row
    yrow = torch.cat([torch.zeros(1, dtype=f64, device=dev), torch.cumsum(dy, 0)])
    i = torch.arange(nx + 1, dtype=f64, device=dev)
    jit = torch.rand((2, nx + 1, ny), generator=g, dtype=f64, device=dev) * 0.7 - 0.35
    xcol = (10.0 - torch.sqrt(100.0 - 99.0 * i / nx)) / 9.0
    dx = torch.cat([xcol[1:2] - xcol[:1], torch.minimum(xcol[2:] - xcol[1:-1], xcol[1:-1] - xcol[:-2]),
                    xcol[-1:] - xcol[-2:-1]])
    reach = torch.minimum(dx[:, None], ly[None, :])
    X = xcol[:, None] + jit[0] * reach
    Y = yrow[None, :] + jit[1] * reach

    def cot(p, q, r):       # cotangent at p of the triangle p q r
        ux, uy, vx, vy = q[0] - p[0], q[1] - p[1], r[0] - p[0], r[1] - p[1]
        return (ux * vx + uy * vy) / torch.clamp((ux * vy - uy * vx).abs(), min=1e-300)

    A, B = (X[:-1, :-1], Y[:-1, :-1]), (X[1:, :-1], Y[1:, :-1])
    C, D = (X[1:, 1:], Y[1:, 1:]), (X[:-1, 1:], Y[:-1, 1:])
    s = cot(B, A, C) + cot(D, A, C) >= 0.0          # Delaunay choice of the quad's diagonal: A-C, else B-D
    zero = torch.zeros((), dtype=f64, device=dev)
    E = torch.zeros((nx + 1, ny), dtype=f64, device=dev)     # (i, j) - (i + 1, j)
    N = torch.zeros_like(E)                                   # (i, j) - (i, j + 1)
    E[:-1, :-1] += torch.where(s, cot(C, A, B), cot(D, A, B))
    E[:-1, 1:] += torch.where(s, cot(A, C, D), cot(B, C, D))
    N[:-1, :-1] += torch.where(s, cot(C, A, D), cot(B, A, D))
    N[1:, :-1] += torch.where(s, cot(A, B, C), cot(D, B, C))
    AC = torch.where(s, cot(B, A, C) + cot(D, A, C), zero)
    BD = torch.where(s, zero, cot(A, B, D) + cot(C, B, D))
    E, N, AC, BD = (0.5 * torch.clamp(w, min=0.0) for w in (E, N, AC, BD))
    Wt = torch.zeros((nx + 1, ny, 9), dtype=f64, device=dev)   # slot 3 (di + 1) + (dj + 1)
    Wt[1:, 1:, 0] = AC
    Wt[1:, :, 1] = E[:-1]
    Wt[1:, :-1, 2] = BD
    Wt[:, 1:, 3] = N[:, :-1]
    Wt[:, :-1, 5] = N[:, :-1]
    Wt[:-1, 1:, 6] = BD
    Wt[:-1, :, 7] = E[:-1]
    Wt[:-1, :-1, 8] = AC
    Wt = torch.where(Wt > 1e-12 * Wt.amax(2, keepdim=True), Wt, zero)
    keep = Wt > 0.0
    # symmetric pattern: an edge is kept if both ends keep it
    for k, di, dj in ((0, -1, -1), (1, -1, 0), (2, -1, 1), (3, 0, -1)):
        o = 8 - k
        src = keep[max(0, -di):nx + 1 - max(0, di), max(0, -dj):ny - max(0, dj), k]
        dst = keep[max(0, di):nx + 1 + min(0, di), max(0, dj):ny + min(0, dj), o]
        both = src & dst
        src.copy_(both)
        dst.copy_(both)
    diag = torch.where(keep, Wt, zero).sum(2)
    Wt = -Wt
    Wt[..., 4] = diag
    keep[..., 4] = True
    keep[nx - 1, :, 6:] = False                               # couplings to the Dirichlet column stay on the diagonal
    Wt, keep = Wt[:nx].reshape(-1, 9), keep[:nx].reshape(-1, 9)
    rows = torch.arange(nx * ny, device=dev)
    off = torch.tensor([di * ny + dj for di in (-1, 0, 1) for dj in (-1, 0, 1)], device=dev)
    return _slots_to_csr(rows[:, None] + off[None, :], Wt, keep)


def _grid(n, dim, seed):
    m = max(4, int(round(n ** (1.0 / dim))))
    dev, f64 = "cuda", torch.float64
    u = torch.rand(2 + dim, generator=_gen(seed), dtype=f64, device=dev).cpu().tolist()
    ratio, radius = 10.0 ** (-1.0 - 2.0 * u[0]), 0.1 + 0.2 * u[1]
    x = (torch.arange(m, dtype=f64, device=dev) + 1) / (m + 1)
    d2 = 0.0
    for a in range(dim):
        shape = [1] * dim
        shape[a] = m
        d2 = d2 + (x.reshape(shape) - (0.35 + 0.3 * u[2 + a])) ** 2
    k = torch.where(d2 < radius ** 2, torch.full_like(d2, ratio), torch.ones_like(d2))
    idx = torch.arange(m ** dim, device=dev).reshape([m] * dim)
    diag = torch.zeros_like(k)
    slots = {}
    for a in range(dim):
        k0, k1 = k.narrow(a, 0, m - 1), k.narrow(a, 1, m - 1)
        face = 2.0 * k0 * k1 / (k0 + k1)
        stride = m ** (dim - 1 - a)
        lo, hi = torch.zeros_like(k), torch.zeros_like(k)
        hi.narrow(a, 0, m - 1).copy_(face)
        lo.narrow(a, 1, m - 1).copy_(face)
        slots[-stride], slots[stride] = -lo, -hi
        diag = diag + lo + hi
        diag.narrow(a, 0, 1).add_(k.narrow(a, 0, 1))           # Dirichlet faces
        diag.narrow(a, m - 1, 1).add_(k.narrow(a, m - 1, 1))
    slots[0] = diag
    offs = sorted(slots)
    vals = torch.stack([slots[o].reshape(-1) for o in offs], 1)
    cols = idx.reshape(-1)[:, None] + torch.tensor(offs, device=dev)[None, :]
    return _slots_to_csr(cols, vals, vals != 0.0)


def _matrix(case, seed, n=None):
    n = case["n"] if n is None else n
    if case["mesh"] == "fv":
        return W.fv_mesh("graded", n, seed)[0]
    if case["mesh"] == "tri":
        return _tri(n, case.get("aspect", 1), seed)
    return _grid(n, 2 if case["mesh"] == "grid2" else 3, seed)


def _rhs(seed, n):
    """Zero-mean U[-1, 1) right-hand side."""
    b = torch.rand(n, generator=_gen(seed + 7919), dtype=torch.float64, device="cuda") * 2.0 - 1.0
    return b - b.mean()


# ----------------------------------------------------------------------------
# prepare / run
# ----------------------------------------------------------------------------
class _Context:
    """An amg context that goes with its owner."""

    def __init__(self, **options):
        self.h = P.amg_create(**options)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            P.amg_destroy(self.h)
            self.h = None


class _Trainer:
    def __init__(self, theta, precision):
        self.h = P.gcin_trainer_create(theta, precision=precision)

    def __del__(self):
        if getattr(self, "h", None) is not None:
            P.gcin_trainer_destroy(self.h)
            self.h = None


def _theta(case):
    """The committed parameters for the mesh kind and network width."""
    h32 = case.get("hidden", 64) == 32
    if case["mesh"] in ("tri", "fv"):
        name = "gcin_c3_h32.npy" if h32 else "gcin_wide.npy"
    else:
        name = "gcin_struct_h32.npy" if h32 else "gcin_struct.npy"
    return np.load(os.path.join(WEIGHTS, name)).astype(np.float32)


def _coeffs(case, n_levels):
    return np.tile(np.asarray(COEFFS[case["mesh"]]), (n_levels, 1))


def _context(case, A):
    ctx = _Context(precision=P.AMG_FP64 if case.get("precision") == "fp64" else P.AMG_FP32_IN_FP64,
                   outer=P.AMG_OUTER_PCG if case.get("outer") == "pcg" else P.AMG_OUTER_REFINE,
                   gnn_precision=P.AMG_GNN_FP32 if case.get("net") == "fp32" else P.AMG_GNN_BF16,
                   max_levels=16)
    if case["setup"] == "device":
        P.amg_setup_device(ctx.h, A, 0, P.AMG_SPLIT_RS_BLOCKS)
    else:
        P.amg_setup(ctx.h, A)
    return ctx


def _batch_sizes(case):
    k = case.get("batch", 1)
    return [max(500, int(case["n"] * (0.5 + t / max(1, k - 1)))) if k > 1 else case["n"] for t in range(k)]


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case}
    if op in ("loss", "train"):
        sizes = _batch_sizes(case)
        mats = [_matrix(case, seed * 16 + k, n) for k, n in enumerate(sizes)]
        s["ctxs"] = [_context(case, A) for A in mats]
        s["f"] = [_rhs(seed * 16 + k, A.n_rows).cpu().numpy() for k, A in enumerate(mats)]
        s["n_vc"] = case["n_vc"]
        if op == "loss":
            c = _coeffs(case, P.amg_num_levels(s["ctxs"][0].h)).astype(np.float32)
            s["c"] = torch.from_numpy(c).requires_grad_(True)
        else:
            th = _theta(case)
            s["theta"] = torch.from_numpy(th).requires_grad_(True)
            s["trainer"] = _Trainer(th, P.AMG_GNN_FP32 if case["net"] == "fp32" else P.AMG_GNN_BF16)
            s["levels"] = [P.amg_num_levels(c.h) for c in s["ctxs"]]
        return s
    A = _matrix(case, seed)
    s["ctx"] = _context(case, A)
    if op in ("predict", "step"):
        P.gnn_load_params(s["ctx"].h, _theta(case))
    elif case["smoother"] == "gnn":
        P.amg_set_coeffs(s["ctx"].h, _coeffs(case, P.amg_num_levels(s["ctx"].h)))
    if op != "predict":
        s["b"] = _rhs(seed, A.n_rows)
    if op == "vcycle":
        s["e"] = torch.empty_like(s["b"])
    return s


def _solve(s):
    x = torch.zeros_like(s["b"])
    status, _ = P.amg_solve_device(s["ctx"].h, s["b"], x, 1e-8)
    return {"x": x, "status": int(status)}


def run(s):
    op = s["op"]
    if op == "solve":
        return _solve(s)
    if op == "step":
        c = P.gnn_predict_coeffs(s["ctx"].h)
        return {"c": c.astype(np.float32), **_solve(s)}
    if op == "predict":
        return {"c": P.gnn_predict_coeffs(s["ctx"].h).astype(np.float32)}
    if op == "vcycle":
        P.amg_vcycle_device(s["ctx"].h, s["b"], s["e"])
        return {"e": s["e"] if s["case"]["precision"] == "fp64" else s["e"].float()}
    if op == "loss":
        s["c"].grad = None
        L = AG.gnn_amg_loss(s["c"], s["ctxs"][0].h, s["f"][0], s["n_vc"])
        L.backward()
        return {"loss": L.detach(), "dc": s["c"].grad}
    s["theta"].grad = None
    c = AG.gcin_coefficients(s["theta"], s["trainer"].h, [x.h for x in s["ctxs"]])
    L, row = 0.0, 0
    for ctx, f, nl in zip(s["ctxs"], s["f"], s["levels"]):
        L = L + AG.gnn_amg_loss(c[row:row + nl], ctx.h, f, s["n_vc"]) / (s["n_vc"] * len(s["ctxs"]))
        row += nl
    L.backward()
    return {"loss": L.detach(), "c": c.detach(), "dtheta": s["theta"].grad}


# ----------------------------------------------------------------------------
# the work no implementation can do without
# ----------------------------------------------------------------------------
def _finest(case, n):
    if case["mesh"] in ("tri", "fv"):
        return n, 7 * n
    d = 2 if case["mesh"] == "grid2" else 3
    m = max(4, int(round(n ** (1.0 / d))))
    return m ** d, (2 * d + 1) * m ** d


def work(case):
    """Each level's matrices read once and its vectors read and written once
    (all levels together: about 1.9 times the finest one's entries); a solve
    once per pass in all (its cycle count is the method's), the network's
    activations once."""
    op = case["op"]
    tb = 8 if case.get("precision") == "fp64" else 4
    out = {"bytes": 0.0, "flops": 0.0}
    for n in _batch_sizes(case) if op in ("loss", "train") else [case["n"]]:
        n, nnz = _finest(case, n)
        n_all, nnz_all = 1.65 * n, 1.9 * nnz
        cycle_bytes = (tb + 4.0) * nnz_all * 1.5 + 3.0 * tb * n_all
        cycle_flops = 2.0 * nnz_all * (9.0 if case.get("smoother", "gnn") == "gnn" else 5.0)
        H = case.get("hidden", 64)
        net_bytes = 8.0 * nnz_all + 4 * 2 * (2.0 if case.get("net") == "bf16" else 4.0) * H * n_all
        net_flops = 3 * (2.0 * nnz_all * H + 2.0 * n_all * H * H)
        if op in ("vcycle", "solve", "step"):
            out["bytes"] += cycle_bytes + 16.0 * n
            out["flops"] += cycle_flops
        if op in ("predict", "step"):
            out["bytes"] += net_bytes
            out["flops"] += net_flops
        if op in ("loss", "train"):
            out["bytes"] += case["n_vc"] * 3.0 * cycle_bytes
            out["flops"] += case["n_vc"] * 3.0 * cycle_flops
        if op == "train":
            out["bytes"] += 3.0 * net_bytes
            out["flops"] += 3.0 * net_flops
    return out


# ----------------------------------------------------------------------------
# 64-bit results in plain torch (the hierarchy is read back as given input)
# ----------------------------------------------------------------------------
class _Csr:
    def __init__(self, d, ncol):
        self.n, self.ncol = int(d["n"]), ncol
        rp = torch.from_numpy(d["row_ptr"].astype(np.int64)).cuda()
        self.row = torch.repeat_interleave(torch.arange(self.n, device="cuda"), rp[1:] - rp[:-1])
        self.col = torch.from_numpy(d["col"].astype(np.int64)).cuda()
        self.val = torch.from_numpy(d["val"]).cuda()

    def mv(self, x, val=None):
        v = self.val if val is None else val
        y = torch.zeros((self.n,) + x.shape[1:], dtype=x.dtype, device=x.device)
        w = v if x.dim() == 1 else v[:, None]
        return y.index_add(0, self.row, w * x[self.col])

    def tmv(self, x):
        y = torch.zeros(self.ncol, dtype=x.dtype, device=x.device)
        return y.index_add(0, self.col, self.val * x[self.row])


class _Level:
    def __init__(self, ctx, l):
        a, p = P.amg_get_level(ctx, l)
        self.A = _Csr(a, int(a["n"]))
        self.P = None if p is None else _Csr(p, int(p["nc"]))
        on = self.A.row == self.A.col
        self.on = on
        self.diag = torch.zeros(self.A.n, dtype=torch.float64, device="cuda").index_add(0, self.A.row[on],
                                                                                          self.A.val[on])
        off = self.A.val[~on].abs()
        self.s = off.max() if off.numel() else torch.ones((), dtype=torch.float64, device="cuda")

    def q(self, c):
        """Pseudo-inverse values on A's pattern from (d0, d1, d2, o1, o2)."""
        x = self.A.val / self.s
        den = torch.where(self.on, self.diag[self.A.row], self.diag[self.A.row] + self.diag[self.A.col])
        return torch.where(self.on, c[0] + c[1] * x + c[2] * x * x, c[3] * x + c[4] * x * x) / den


def _levels(ctx):
    return [_Level(ctx, l) for l in range(P.amg_num_levels(ctx))]


def _cycle(levels, l, b, qs, dense):
    L = levels[l]
    if l == len(levels) - 1:
        return torch.cholesky_solve(b[:, None], dense)[:, 0]

    def sweep(u):
        r = b - L.A.mv(u)
        return u + (L.A.mv(r, qs[l]) if qs is not None else OMEGA * r / L.diag)

    u = L.A.mv(b, qs[l]) if qs is not None else OMEGA * b / L.diag
    u = sweep(u)
    e = _cycle(levels, l + 1, L.P.tmv(b - L.A.mv(u)), qs, dense)
    return sweep(sweep(u + L.P.mv(e)))


def _dense(levels):
    L = levels[-1].A
    M = torch.zeros((L.n, L.n), dtype=torch.float64, device="cuda")
    M.index_put_((L.row, L.col), L.val, accumulate=True)
    return torch.linalg.cholesky(M)


def _exact_x(levels, b):
    """A^-1 b by conjugate gradients with the Jacobi V-cycle, refined."""
    dense, A = _dense(levels), levels[0].A
    x = torch.zeros_like(b)
    for _ in range(3):
        r0 = r = b - A.mv(x)
        d, p, rz = torch.zeros_like(b), None, None
        for _ in range(200):
            z = _cycle(levels, 0, r, None, dense)
            new = torch.dot(r, z)
            p = z if p is None else z + (new / rz) * p
            rz = new
            q = A.mv(p)
            a = rz / torch.dot(p, q)
            d, r = d + a * p, r - a * q
            if float(r.norm()) <= 1e-9 * float(r0.norm()):
                break
        x = x + d
    return x


def _exact_net(theta, levels):
    """Coefficients of every level graph from the flat parameters."""
    H = 64 if theta.numel() == P.AMG_GCIN_NUM_PARAMS else 32
    shapes = [(2, H), (H,)] + [(H, H), (H,)] * 3 + [(H,), (H,)] * 4 + [(2 * H, 32), (32,)] * 4 + [(128,), (128,)]
    shapes += [(128, 128), (128,), (128, 64), (64,), (64, 5), (5,)]
    t, o = [], 0
    for sh in shapes:
        k = int(np.prod(sh))
        t.append(theta[o:o + k].reshape(sh))
        o += k
    out = []
    for L in levels:
        deg = torch.zeros_like(L.diag).index_add(0, L.A.row[~L.on], torch.ones_like(L.A.val[~L.on]))
        x = torch.stack([L.diag, deg], 1)
        z = []
        for k in range(4):
            y = L.A.mv(x) @ t[2 * k] + t[2 * k + 1]
            y = (y - y.mean(0)) / torch.sqrt(y.var(0, unbiased=False) + 1e-5)
            x = torch.relu(y * t[8 + 2 * k] + t[9 + 2 * k])
            z.append(torch.cat([x.mean(0), x.max(0).values]) @ t[16 + 2 * k] + t[17 + 2 * k])
        z = torch.cat(z)
        z = (z - z.mean()) / torch.sqrt(z.var(unbiased=False) + 1e-5) * t[24] + t[25]
        z = torch.relu(torch.sigmoid(z) @ t[26] + t[27])
        out.append(torch.relu(z @ t[28] + t[29]) @ t[30] + t[31])
    return torch.stack(out)


def _exact_loss(levels, c, f, n_vc):
    dense, A = _dense(levels), levels[0].A
    qs = [L.q(c[l]) for l, L in enumerate(levels[:-1])]
    u = torch.zeros_like(f)
    for _ in range(n_vc):
        u = u + _cycle(levels, 0, f - A.mv(u), qs, dense)
    return torch.log10(torch.linalg.vector_norm(f - A.mv(u)) / torch.linalg.vector_norm(f))


def exact(case, seed):
    s = prepare(case, seed)
    op = case["op"]
    if op in ("loss", "train"):
        levels = [_levels(c.h) for c in s["ctxs"]]
        fs = [torch.from_numpy(f).cuda() for f in s["f"]]
        if op == "loss":
            c = s["c"].detach().double().cuda().requires_grad_(True)
            L = _exact_loss(levels[0], c, fs[0], case["n_vc"])
            L.backward()
            return {"loss": L.detach(), "dc": c.grad}
        th = s["theta"].detach().double().cuda().requires_grad_(True)
        c = _exact_net(th, [lv for ls in levels for lv in ls])
        total, row = 0.0, 0
        for ls, f in zip(levels, fs):
            total = total + _exact_loss(ls, c[row:row + len(ls)], f, case["n_vc"]) / (case["n_vc"] * len(fs))
            row += len(ls)
        total.backward()
        return {"loss": total.detach(), "c": c.detach(), "dtheta": th.grad}
    levels = _levels(s["ctx"].h)
    out = {}
    if op in ("predict", "step"):
        with torch.no_grad():
            out["c"] = _exact_net(torch.from_numpy(_theta(case)).double().cuda(), levels)
    if op in ("solve", "step"):
        out.update(x=_exact_x(levels, s["b"]), status=None)
    if op == "vcycle":
        qs = None
        if case["smoother"] == "gnn":
            qs = [L.q(COEFFS[case["mesh"]]) for L in levels[:-1]]
        out["e"] = _cycle(levels, 0, s["b"], qs, _dense(levels))
    return out
