"""Row sums of the learned-SPAI network where rows are cut by the 32-edge ranges of the
message layer's warps: rows of one edge, rows that begin or end at a cut, rows over many
cuts, more cut edges than one batch of the node update (16), and a last range that is not
full.  Inference (which stores only the messages behind a cut) and the loss (which stores
all) against the float64 oracle.

Tolerance: a float32 sum of k messages, taken in order, is off by at most k 2^-24 of the sum
of their sizes, 1.2e-5 at the 200 edges a row used here; four layers and the decoder follow,
and the products' operands are split to below 2^-21, so 1e-4 of the largest entry of M, and
of the loss, covers them."""
import numpy as np
import pytest
import scipy.sparse as sp

import synth
from oracle import gnn as ognn

pytestmark = pytest.mark.gpu


def _matrix(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "diagonal":                              # one edge a row, no cuts
        M = sp.eye(n, format="lil")
    elif kind == "arrow":                               # one row over many cuts, short ones
        M = sp.eye(n, format="lil")
        M[n // 2, :] = rng.standard_normal(n)
        M[:, n // 2] = rng.standard_normal((n, 1))
    else:                                               # rows of 1 .. about 2 * mean edges
        mean = int(kind)
        M = sp.lil_matrix((n, n))
        for i in range(n):
            c = rng.integers(0, n, rng.integers(0, mean + 1))
            M[i, c] = rng.standard_normal(len(c))
        M = (M + M.T).tolil()
    M = M.tocsr()
    M.setdiag(4.0 + rng.random(n))
    M.sort_indices()
    return synth.CSR.from_scipy(M)


@pytest.mark.parametrize("kind,n", [("diagonal", 1), ("diagonal", 33), ("arrow", 200), ("3", 257),
                                    ("16", 300), ("31", 128), ("90", 150)])
def test_cut_rows_match_oracle(rbo, kind, n):
    import torch
    A = _matrix(kind, n, 7)
    G = ognn.Graph(A)
    rng = np.random.default_rng(3)
    th = ognn.init_params(5)
    th[-97:] = rng.standard_normal(97) * 0.05
    th = th.astype(np.float32)
    net = rbo.GNN(seed=0)
    net.set_params(th)
    Ad = rbo.DeviceCSR.from_host(A)
    M = net.infer(Ad).cpu().numpy()
    ref = ognn.forward(th.astype(np.float64), G, bf16=True)
    assert np.abs(M - ref).max() <= 1e-4 * np.abs(ref).max()
    R = rng.standard_normal((n, 4))
    Rd = rbo.colmajor(n, 4)
    Rd.copy_(torch.from_numpy(R))
    L, _ = net.loss_grad(Ad, Rd)
    Lr, _ = ognn.loss_and_grad(th.astype(np.float64), G, R, bf16=True)
    assert abs(L - Lr) <= 1e-4 * abs(Lr)
