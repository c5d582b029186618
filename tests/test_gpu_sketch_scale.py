"""Scales of the sketch's integer sums: values at the top of the float64 range, outliers, and
columns that fall over the rows.  4096 x 3 sums of 8 bytes leave room for one CTA per SM, so that
CTA i of 152 takes the tiles i, i + 152, .. of 64 rows."""
import numpy as np
import pytest

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

CTAS = 152


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_after_the_largest_finite_value(rbo, bad):
    """A value of 2^1023 puts the column's scale at its top before the same CTA meets the
    non-finite value."""
    n = 200000
    W = np.zeros((n, 3))
    W[0] = 2.0 ** 1023
    W[CTAS * 64 + 7, 1] = bad
    out = rbo.sketch_apply(rbo.sketch_create(n, 4096, 8, 42), to_dev(W))
    assert np.isnan(out[:, 1]).all()
    assert not np.isnan(out[:, [0, 2]]).any()


@pytest.mark.parametrize("n,k,zeta", [(400001, 3, 1), (200000, 3, 2)])
def test_outliers_cost_other_tiles_nothing(rbo, n, k, zeta):
    """Values of 1e12 in the first tile of every CTA, then of 1, and a column that falls by 2^-40
    over the rows: a value is rounded at 2^-46 of the largest of its own tile of at most 64 rows
    at worst (half a unit of 2^-53 of a scale whose exponent may lie 8 above that), the sums of a
    tile are exact, and the float64 sums over flushes, CTAs and groups are at most 2048
    additions."""
    d = 4096
    rng = np.random.default_rng(n)
    W = rng.standard_normal((n, k))
    W[0:CTAS * 64:64, :k - 1] *= 1e12
    W[:, k - 1] *= 2.0 ** (-40.0 * np.arange(n) / n)
    sk = rbo.sketch_create(n, d, zeta, 42)
    got = rbo.sketch_apply(sk, to_dev(W))
    idx, sg = (t.cpu().numpy().reshape(n, zeta) for t in rbo.sketch_entries(sk, 0, n))
    nt = (n + 63) // 64
    top = np.abs(np.pad(W, ((0, 64 * nt - n), (0, 0)))).reshape(nt, 64, k).max(axis=1)
    top = np.repeat(top, 64, axis=0)[:n]
    ref = np.zeros((d, k), dtype=np.longdouble)
    unit, size = np.zeros((d, k)), np.zeros((d, k))
    for j in range(zeta):
        np.add.at(ref, idx[:, j], sg[:, j][:, None] * W.astype(np.longdouble))
        np.add.at(unit, idx[:, j], top)
        np.add.at(size, idx[:, j], np.abs(W))
    bound = 2.0 ** -46 * unit + 2048 * 2.0 ** -53 * size
    assert (np.abs(got - ref) <= bound).all()
