"""The SpMV of short rows stages 256 rows a block with bulk copies: row counts around the
block, empty rows, a block with more entries than the staging holds, pieces that start and
end anywhere in a 16-byte group, and index and value arrays that are not 16-byte aligned
(read from global memory instead), with and without a column scale.

Tolerance: a row of k entries is two chains of fused operations and one addition, off by at
most (k + 2) 2^-53 of the sum of the sizes of its terms (scaling adds one rounding a term)."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,long_row,shift,scale", [(1, 0, 0, False), (255, 0, 0, True), (256, 0, 1, False),
                                                    (257, 0, 0, False), (1000, 900, 0, True),
                                                    (1000, 900, 1, False), (5003, 0, 0, False)])
def test_short_rows_match_scipy(rbo, n, long_row, shift, scale):
    import torch
    rng = np.random.default_rng(n + shift)
    rows, cols = [], []
    for i in range(n):
        c = np.unique(rng.integers(0, n, rng.integers(0, 8)))
        if long_row and i == n // 3:
            c = np.arange(long_row)
        rows += [i] * len(c)
        cols += list(c)
    M = sp.csr_matrix((rng.standard_normal(len(rows)), (rows, cols)), shape=(n, n))
    A = rbo.DeviceCSR(n, M.indptr, M.indices, M.data)
    if shift:
        col = torch.zeros(A.nnz + 1, dtype=torch.int32, device="cuda")
        val = torch.zeros(A.nnz + 1, dtype=torch.float64, device="cuda")
        col[1:], val[1:] = A.col, A.val
        A.col, A.val = col[1:], val[1:]
    x = rng.standard_normal(n)
    d = rng.uniform(0.5, 2.0, n) if scale else np.ones(n)
    ds = torch.from_numpy(d).cuda() if scale else None
    y = rbo.mpk_csr(A, torch.from_numpy(x).cuda(), 1, dscale=ds)[:, 0].cpu().numpy()
    ref = M @ (d * x)
    size = abs(M) @ np.abs(d * x)
    k = np.diff(M.indptr)
    assert (np.abs(y - ref) <= 2 * (k + 3) * 2.0 ** -53 * size).all()
