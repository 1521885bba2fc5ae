"""The network's reductions (instance-norm statistics, pooling) past FP32's range.

Large entries square in the features and again in the variance, so a graph's
sum can leave FP32's range while its parts, its mean or the normalised
features stay inside it.  Each case scales a layer's parameters so that the
exact result is known from the unscaled network:
* a layer's linear by 2^70: every variance overflows FP32, 1 / std is zero and
  the layer's features are ReLU(beta), as with gamma = 0: the same bits;
* layer 1 such that only the finest graph's sum of squares overflows, no
  chunk's of it: the instance norm removes the factor (bar 1e-5, the FP32 network's; the factor
  is no power of two);
* the last layer's gamma and beta by 2^k and its readout rows by 2^-k, with
  the graph's (k = 116) or every tile's (k = 121) sum past the range: the
  coefficients are unchanged (bar 1e-6: roundings of the pooled means, and of
  the smallest readout rows, which leave the normal range).
"""
import numpy as np
import pytest

import paper_2606_19251_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu

FLT_MAX = float(np.finfo(np.float32).max)


def _slices(H):
    """Flat parameter vector: slices of conv W/b, norm gamma/beta, readout W/b per layer."""
    sizes = [n for l in range(4) for n in ((2 if l == 0 else H) * H, H)] + [H] * 8 + [2 * H * 32, 32] * 4
    ends = np.cumsum(sizes)
    s = [slice(int(e) - n, int(e)) for e, n in zip(ends, sizes)]
    return s[0:8:2], s[1:8:2], s[8:16:2], s[9:16:2], s[16::2]


@pytest.fixture(scope="module")
def mesh():
    return W.fv_mesh("graded", 30000, 3)[0]


def _predict(A, net, thetas):
    ctx = P.amg_create(gnn_precision=net)
    try:
        P.amg_setup(ctx, A)
        out = []
        for th in thetas:
            P.gnn_load_params(ctx, th.astype(np.float32))
            out.append(P.gnn_predict_coeffs(ctx))
        return out
    finally:
        P.amg_destroy(ctx)


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("net", [P.AMG_GNN_FP32, P.AMG_GNN_BF16])
@pytest.mark.parametrize("H", [64, 32])
def test_overflowing_variance_leaves_beta(mesh, H, net):
    W_, b_, ga, be, _ = _slices(H)
    base = W.gcin_init_params(5, last_scale=1.0, hidden=H)
    for l in range(4):
        base[be[l]] = np.random.default_rng(l).normal(size=H)
        big, zero = base.copy(), base.copy()
        big[W_[l]] *= 2.0 ** 70
        big[b_[l]] *= 2.0 ** 70
        zero[ga[l]] = 0.0
        got, want = _predict(mesh, net, [big, zero])
        assert np.array_equal(got, want), l


@pytest.mark.parametrize("H", [64, 32])
def test_only_the_graph_sum_of_squares_overflows(mesh, H):
    W_, b_, _, _, _ = _slices(H)
    base = W.gcin_init_params(6, last_scale=1.0, hidden=H)
    n, rp, col, val = mesh.n_rows, np.asarray(mesh.row_ptr), np.asarray(mesh.col), np.asarray(mesh.val)
    row = np.repeat(np.arange(n), np.diff(rp))
    x = np.stack([np.bincount(row[row == col], val[row == col], n), np.diff(rp) - 1.0], 1)
    h = np.stack([np.bincount(row, val * x[col, k], n) for k in range(2)], 1)
    y = h @ base[W_[0]].reshape(2, H) + base[b_[0]]
    total = ((y - y.mean(0)) ** 2).sum(0)
    # chunks are runs of 64 tiles of 64 nodes on a mesh of this size
    chunk = max(((y[i:i + 4096] - y[i:i + 4096].mean(0)) ** 2).sum(0).max() for i in range(0, n, 4096))
    assert total.max() > 1.5 * chunk
    a = np.sqrt(FLT_MAX / np.sqrt(total.max() * chunk))     # total a^2 > FLT_MAX > chunk a^2
    small, big = base.copy(), base.copy()
    for th, s in ((small, a * 2.0 ** -30), (big, a)):
        th[W_[0]] *= s
        th[b_[0]] *= s
    want, got = _predict(mesh, P.AMG_GNN_FP32, [small, big])
    # the finest graph's row: on the coarser graphs, of one chunk, the chunk overflows
    assert _rel(got[0], want[0]) < 1e-5


@pytest.mark.parametrize("net", [P.AMG_GNN_FP32, P.AMG_GNN_BF16])
@pytest.mark.parametrize("H", [64, 32])
@pytest.mark.parametrize("k", [116, 121])
def test_pooled_sums_past_the_range(mesh, H, k, net):
    _, _, ga, be, ro = _slices(H)
    base = W.gcin_init_params(7, last_scale=1.0, hidden=H)
    base[ga[3]] = 0.1
    base[be[3]] = 3.0
    big = base.copy()
    for s in (ga[3], be[3]):
        big[s] *= 2.0 ** k
    big[ro[3]] *= 2.0 ** -k
    want, got = _predict(mesh, net, [base, big])
    assert _rel(got, want) < 1e-6
