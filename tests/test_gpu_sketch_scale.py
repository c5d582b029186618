"""Scales of the sketch's integer sums: values at the top of the float64 range."""
import numpy as np
import pytest

from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_after_the_largest_finite_values(rbo, bad):
    """Every CTA's first tile holds a value of 2^1023, so that the scale is at its top when the
    non-finite value comes (tiles beyond the first of a CTA: more than 8 x 152 tiles of 64 rows)."""
    n = 200000
    W = np.zeros((n, 2))  # (the sums of column 1 overflow)
    W[0:1216 * 64:64] = 2.0 ** 1023
    W[1216 * 64 + 1000, 0] = bad
    out = rbo.sketch_apply(rbo.sketch_create(n, 40, 8, 42), to_dev(W))
    assert np.isnan(out[:, 0]).all()
