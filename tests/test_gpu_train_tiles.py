"""The FP32 network backward at the edges of its 64-node tiles: graphs one node
short of a tile, whole tiles, one node past them and a batch of all of them,
for both widths, against autograd through the oracle's network.  Bar: the
network backward's 1e-4 of the gradient's norm."""
import numpy as np
import pytest
import torch
from scipy.sparse import csr_matrix
from scipy.sparse.csgraph import reverse_cuthill_mckee

import paper_2606_19251_gb300 as P
import workloads as W
from oracle import gcin as OG
from oracle import setup as OS
from tests.gpu_helpers import ctx_setup

pytestmark = pytest.mark.gpu

SIZES = [63, 64, 65, 127, 128, 129]


def _leading(A, n):
    """Leading n x n block of a mesh matrix in RCM order (a connected strip,
    still an M-matrix)."""
    M = csr_matrix((np.asarray(A.val), np.asarray(A.col), np.asarray(A.row_ptr)), shape=(A.n_rows, A.n_rows))
    place = np.empty(A.n_rows, dtype=np.int64)
    place[reverse_cuthill_mckee(M, symmetric_mode=True)] = np.arange(A.n_rows)
    rows = place[np.repeat(np.arange(A.n_rows), np.diff(A.row_ptr))]
    cols = place[np.asarray(A.col, dtype=np.int64)]
    keep = (rows < n) & (cols < n)
    return W._coo_to_csr(n, n, rows[keep], cols[keep], np.asarray(A.val)[keep])


@pytest.mark.parametrize("hidden", [64, 32])
@pytest.mark.parametrize("sizes", [[n] for n in SIZES] + [SIZES])
def test_backward_at_tile_edges(sizes, hidden):
    mesh = W.fv_mesh("graded", 2000, 3)[0]
    mats = [_leading(mesh, n) for n in sizes]
    theta = W.gcin_init_params(11, last_scale=1.0, hidden=hidden)
    ctxs = [ctx_setup(A, P.AMG_FP32_IN_FP64, max_coarse=256) for A in mats]      # one level each
    tr = P.gcin_trainer_create(theta, precision=P.AMG_GNN_FP32)
    try:
        assert [P.amg_num_levels(c) for c in ctxs] == [1] * len(sizes)
        c = P.gcin_trainer_forward(tr, ctxs)
        dc = np.random.default_rng(0).standard_normal(c.shape)
        g = P.gcin_trainer_backward(tr, dc)
        graphs = [OG.Graph(OS.build_hierarchy(A, max_coarse=256)[0].A) for A in mats]
        t = torch.tensor(np.asarray(theta, dtype=np.float32).astype(np.float64), requires_grad=True)
        cref = OG.forward(t, graphs)
        (cref * torch.from_numpy(dc)).sum().backward()
        gref = t.grad.numpy()
        assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    finally:
        P.gcin_trainer_destroy(tr)
        for c_ in ctxs:
            P.amg_destroy(c_)
