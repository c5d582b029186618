"""Passes of few columns over many rows run on the float64 pipe, the others on the tensor cores:
both sides of that line, aligned and not, rows that leave a ragged tile, against the oracle.

Tolerances: a float64 sum of n products is off by at most n 2^-53 of the sum of their sizes in
any order, and a digit product by 2^-50 of the largest product of its chunk of at most 128 rows
a term (as in the tests of tall tiles); Q and R of a well-conditioned V as elsewhere."""
import numpy as np
import pytest

import synth
from oracle import metrics
from oracle.dense import gram as ogram

from test_gpu_tall_tiles import _bound, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [77823, 77825, 100095])
@pytest.mark.parametrize("a,b", [(1, 5), (5, 4), (6, 5), (10, 2), (16, 1), (17, 2), (60, 1), (71, 1), (72, 1), (1, 8)])
def test_gram_on_both_sides(rbo, n, a, b):
    rng = np.random.default_rng(n + 7 * a + b)
    X, Y = rng.standard_normal((n, a)), rng.standard_normal((n, b))
    ref = ogram(X, Y)
    bound = _bound(X, Y) + n * 2.0 ** -53 * (np.abs(X).T @ np.abs(Y))
    assert (np.abs(rbo.gram(_dev(rbo, X), _dev(rbo, Y)) - ref) <= bound).all()
    assert (np.abs(rbo.gram(_dev(rbo, X, n | 1), _dev(rbo, Y, n | 1)) - ref) <= bound).all()


@pytest.mark.parametrize("s,nb", [(1, 7), (2, 5), (3, 4), (4, 3), (5, 2)])
def test_one_stage_of_narrow_blocks(rbo, s, nb):
    n = 78001
    V = synth.glued_blocks(n, nb, s, 10.0, seed=s, v0=True) if s > 1 else \
        np.random.default_rng(1).standard_normal((n, nb + 1))
    sk = rbo.sketch_create(n, 4 * (s * nb + 2), 8, 42)
    R = np.linalg.qr(V, mode="r")
    R *= np.sign(np.diag(R))[:, None]
    for ld in (n + 1, n):
        D = _dev(rbo, V, ld)
        out = rbo.block_orth_one_stage(sk, D, s, v0=True)
        assert metrics.orth_error(D.cpu().numpy()) <= 1e-13
        assert metrics.backward_error(V, D.cpu().numpy(), out.R) <= 1e-14
        assert metrics.rel_diff(out.R, R) <= 1e-12
