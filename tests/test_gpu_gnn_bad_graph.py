"""Matrices whose row pointers or columns do not describe their edges are refused by the
network before anything is read or written by the row or column of an edge."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["edges past the last row", "first row not at 0", "falling", "past the edges",
                                  "negative", "column n", "column -1"])
def test_inconsistent_graph_is_refused(rbo, what):
    P = synth.laplace2d_csr(20)
    rowptr, col, val = P.rowptr.copy(), P.col.copy(), P.val.copy()
    if what == "edges past the last row":
        col, val = np.r_[col, col[:64]], np.r_[val, val[:64]]
    elif what == "first row not at 0":
        rowptr[0] = 2
    elif what == "falling":
        rowptr[200] = rowptr[198] - 1
    elif what == "past the edges":
        rowptr[300] = len(col) + 5
    elif what == "negative":
        rowptr[100] = -3
    else:
        col[77] = P.n if what == "column n" else -1
    A = rbo.DeviceCSR(P.n, rowptr, col, val)
    net = rbo.GNN(seed=0)
    with pytest.raises(rbo.RboError):
        net.infer(A)
    R = rbo.colmajor(P.n, 4)
    R.fill_(1.0)
    with pytest.raises(rbo.RboError):
        net.loss_grad(A, R)
    net.infer(rbo.DeviceCSR.from_host(P))  # the next call is served
