"""Row counts past 2^31, which the coordinates of a tensor copy do not reach (17 GB a column).

The sketch is exact here: integer values, whose sums stay below 2^53.  The norm of the column
is a float64 sum of 2^31 terms, in chains of at most 2^31 / (152 * 256) of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_sketch_and_orthogonalization_of_a_long_column(rbo):
    import torch
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of free device memory")
    n, d, step = (1 << 31) + 77, 24, 1 << 27
    W = rbo.colmajor(n, 1)
    sk = rbo.sketch_create(n, d, 1, 42)
    ref = torch.zeros(d, dtype=torch.float64, device="cuda")
    norm2 = 0
    for r0 in range(0, n, step):
        k = min(step, n - r0)
        W[r0:r0 + k, 0] = (torch.arange(r0, r0 + k, device="cuda") * 7 % 13 - 6).to(torch.float64)
        idx, sg = rbo.sketch_entries(sk, r0, k)
        ref.index_add_(0, idx[:, 0].long(), sg[:, 0].double() * W[r0:r0 + k, 0])
        norm2 += int(W[r0:r0 + k, 0].square().sum())
        del idx, sg
    got = rbo.sketch_apply(sk, W)
    assert np.array_equal(got[:, 0], ref.cpu().numpy())
    out = rbo.block_orth_one_stage(sk, W, 1)
    tol = 2.0 ** 31 / (152 * 256) * 2.0 ** -52
    assert abs(out.R[0, 0] / np.sqrt(norm2) - 1.0) <= tol
    assert abs(float(W[:step, 0].square().sum() + W[step:, 0].square().sum()) - 1.0) <= 2 * tol
    del W
    torch.cuda.empty_cache()
    rbo.release_workspace()
