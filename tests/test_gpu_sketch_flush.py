"""Integer sums of the sparse sketch at the edge of their range.  A sketch row may sum 384
values of up to 2^54 before its sum enters the float64 partial; the entries here are chosen so
that the sums grow as fast as the schedule's counts allow: every value sits at the top of its
column's scale (the first tiles' values are half as large, later ones fill the room that the
scale leaves) and has the sign of its row's first entry.  Few sketch rows (many entries of a
tile in one row, a flush every few tiles) and many.

Tolerance: the integer sums are exact, at most 608 partials are added in float64 (7e-14 of the
sum of the sizes), the reference adds blocks of 1000 rows and then the blocks (at most 2100
terms in a chain, 3e-13); 1e-12 covers both.  An overflow would be off by 2^64 units of 2^-54."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,d,zeta", [(400001, 5, 12, 8), (1100003, 2, 404, 8)])
def test_sums_at_the_top_of_the_scale(rbo, n, k, d, zeta):
    import torch
    sk = rbo.sketch_create(n, d, zeta, 42)
    idx, sg = (t.cpu().numpy() for t in rbo.sketch_entries(sk, 0, n))
    idx, sg = idx.reshape(n, zeta), sg.reshape(n, zeta).astype(np.float64)
    big = np.where(np.arange(n) < 608 * 64, 2.0 - 2.0 ** -52, 4.0 - 2.0 ** -51)
    W = np.stack([sg[:, c % zeta] * big * 2.0 ** (7 * c) for c in range(k)], 1)
    Wd = rbo.colmajor(n, k)
    Wd.copy_(torch.from_numpy(W))
    got = rbo.sketch_apply(sk, Wd)
    ref = np.zeros((d, k))
    size = np.zeros((d, k))
    for r0 in range(0, n, 1000):
        i = idx[r0:r0 + 1000].ravel()
        for c in range(k):
            v = (sg[r0:r0 + 1000] * W[r0:r0 + 1000, c:c + 1]).ravel()
            ref[:, c] += np.bincount(i, v, d)
            size[:, c] += np.bincount(i, np.abs(v), d)
    assert (np.abs(got - ref) <= 1e-12 * size).all()
