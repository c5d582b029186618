"""Gram entries of columns whose large values do not meet: outliers against zeros or small
values, disjoint scales, values that alternate, at shapes of every kind of Gram kernel.

Bound, element by element: a chunk's digits are used where they are off by at most 2^-41 of the
sum of the sizes of its terms, other chunks are sums of float64 products (at most 128 terms);
adding chunks, CTAs and groups rounds once each, at most n / 16 + 1300 times 2^-53."""
import numpy as np
import pytest

from oracle.dense import gram as ogram

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


def _columns(kind, rng, n, c, odd):
    A = rng.standard_normal((n, c))
    r = np.arange(n)
    if kind == "outliers":            # 1e12 in every 64th row of one side, zero there in the other
        A[5::64] *= 0.0 if odd else 1e12
    elif kind == "small there":
        A[5::64] *= 1e-9 if odd else 1e12
    elif kind == "halves":            # large where the other is small, in turn within a chunk
        A *= np.where((r % 2 == 0) == odd, 1.0, 1e-11)[:, None]
    elif kind == "falling":           # one falls and one grows inside every 64 rows
        A *= 2.0 ** ((r % 64) * (-1.0 if odd else 1.0))[:, None]
    elif kind == "one row":
        A[:, 0] = 0.0
        A[n // 2, 0] = 1.0
        A[:, c - 1] = 0.0
        A[n // 3, c - 1] = 3.0
    return A


@pytest.mark.parametrize("kind", ["outliers", "small there", "halves", "falling", "one row"])
@pytest.mark.parametrize("n,a,b", [(1001, 9, 4), (20011, 20, 5), (5003, 40, 16), (8001, 17, 8), (2000, 3, 20)])
def test_gram_elementwise(rbo, kind, n, a, b):
    rng = np.random.default_rng(n + a)
    X, Y = _columns(kind, rng, n, a, False), _columns(kind, rng, n, b, True)
    C = rbo.gram(to_dev(X), to_dev(Y))
    size = np.abs(X).T @ np.abs(Y)
    assert (np.abs(C - ogram(X, Y)) <= (2.0 ** -41 + (n / 16 + 1300 + 128) * 2.0 ** -53) * size).all()


@pytest.mark.parametrize("n", [961, 6403, 6405, 40003])
@pytest.mark.parametrize("s,s_hat", [(5, 30), (10, 50), (16, 16)])
def test_wide_panels_with_a_short_last_tile(rbo, n, s, s_hat):
    """One to five rows in the last tile: some of a panel's entries have small products there, in
    one column tile of a pair and not in the other.  Tolerances as in the other orthogonalization
    tests."""
    import synth
    from gpu_util import to_host
    from oracle import metrics
    V = synth.glued_blocks(n, 2 * s_hat // s, s, 10.0, seed=n, v0=True)
    D = to_dev(V)
    out = rbo.block_orth_two_stage(rbo.sketch_create(n, 4 * (2 * s_hat + 2), 8, 42), D, s, s_hat, v0=True)
    assert metrics.orth_error(to_host(D)) <= 1e-13
    assert metrics.backward_error(V, to_host(D), out.R) <= 1e-14
