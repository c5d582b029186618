"""SpMV of short rows on average where some blocks hold more entries than their staging (entries
staged piece by piece) and some rows are long (summed by a warp, or by the block), aligned or
not, with and without a column scale; a column outside the matrix is reported from each path.

Tolerance: a row of k entries is summed in some fixed order, off by at most (k + 3) 2^-53 of
the sum of the sizes of its terms (a product and a scaling round once each)."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


def _matrix(kind, n, rng):
    k = np.full(n, 2)
    if kind == "dense half":                       # 20 and 2 entries a row: several pieces a block
        k[: n // 2] = 20
    elif kind == "edges":                          # rows at the limits of the three paths
        k[[5, 6, 40, 300, 301, 700, n - 1]] = [128, 129, 4096, 4097, 127, 9000, 5000]
    elif kind == "many":                           # a block of rows longer than a thread walks
        k[256:500] = 200
    M = sp.csr_matrix((np.zeros(k.sum()), np.concatenate([np.sort(rng.choice(n, i, replace=False)) for i in k]),
                       np.concatenate([[0], np.cumsum(k)])), shape=(n, n))
    M.data = rng.standard_normal(M.nnz)
    return M


@pytest.mark.parametrize("kind,n", [("dense half", 2001), ("edges", 12345), ("many", 9001)])
@pytest.mark.parametrize("shift,scale", [(0, False), (1, False), (0, True), (1, True)])
def test_uneven_rows_match_scipy(rbo, kind, n, shift, scale):
    import torch
    rng = np.random.default_rng(n + shift)
    M = _matrix(kind, n, rng)
    assert M.nnz <= 12 * n
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
    size = abs(M) @ np.abs(d * x)
    assert (np.abs(y - M @ (d * x)) <= 2 * (np.diff(M.indptr) + 3) * 2.0 ** -53 * size).all()


@pytest.mark.parametrize("row", [0, 5, 6, 40, 300])
def test_bad_column_is_reported(rbo, row):
    import torch
    n = 12345
    M = _matrix("edges", n, np.random.default_rng(1))
    cols = M.indices.copy()
    cols[M.indptr[row + 1] - 1] = n
    A = rbo.DeviceCSR(n, M.indptr, cols, M.data)
    with pytest.raises(rbo.RboError):
        rbo.mpk_csr(A, torch.ones(n, dtype=torch.float64, device="cuda"), 1)
