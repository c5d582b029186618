"""The largest sketches (rows times panel columns) that the argument checks accept: the dense
step on the sketch then needs nearly all of an SM's shared memory.  One-stage (Householder of
the sketch), two-stage (sketched BCGS2) and the Count-Gauss product, in both precisions that
sketch.

Tolerance: Q and R of a well-conditioned V (kappa = 10) as in the other orthogonalization
tests, 1e-13 and 1e-14."""
import pytest

import synth
from oracle import metrics

from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,nb,s_hat,d,d_inner", [(64, 1, 0, 192, 0), (64, 2, 0, 191, 0), (47, 1, 47, 141, 0),
                                                  (64, 1, 0, 64, 192), (47, 1, 47, 100, 200), (16, 3, 48, 768, 0)])
@pytest.mark.parametrize("precision", ["PREC_FP64", "PREC_MIXED"])
def test_largest_sketches(rbo, s, nb, s_hat, d, d_inner, precision):
    n = 3001
    V = synth.glued_blocks(n, nb, s, 10.0, seed=s + d)
    kind = rbo.SKETCH_COUNT_GAUSS if d_inner else rbo.SKETCH_SPARSE_SIGN
    sk = rbo.sketch_create(n, d, 8, 42, kind, d_inner)
    D = to_dev(V)
    prec = getattr(rbo, precision)
    if s_hat:
        out = rbo.block_orth_two_stage(sk, D, s, s_hat, precision=prec)
    else:
        out = rbo.block_orth_one_stage(sk, D, s, precision=prec)
    Q = to_host(D)
    assert metrics.orth_error(Q) <= 1e-13
    assert metrics.backward_error(V, Q, out.R) <= 1e-14
