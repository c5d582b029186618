"""Row passes with tiles of 128 and 256 rows (from about 39000 and 78000 rows on): ragged last
tiles against the oracle, and arrays that a tensor copy cannot address against aligned ones.

Bound of a digit Gram per chunk of at most 128 rows with largest magnitudes Mx, My: a value is
off by less than 2^-54 of its column's largest, and the digit pairs left out weigh at most
6 * 2^54 / 2^108 < 2^-51.4 of Mx My, so a term is off by less than 2^-50 Mx My; joining a chunk
and adding it round once each, and the float64 sums over chunks and CTAs add at most
(4 chunks) 2^-53 of |X|^T |Y|."""
import numpy as np
import pytest

import synth
from oracle import metrics
from oracle.dense import gram as ogram

pytestmark = pytest.mark.gpu


def _dev(rbo, A, ld=None):
    import torch
    D = rbo.colmajor(*A.shape, ld=ld)
    D.copy_(torch.from_numpy(np.ascontiguousarray(A)))
    return D


def _bound(X, Y):
    n = X.shape[0]
    nt = (n + 127) // 128
    pad = ((0, nt * 128 - n), (0, 0))
    Xa = np.abs(np.pad(X, pad)).reshape(nt, 128, -1).max(axis=1)
    Ya = np.abs(np.pad(Y, pad)).reshape(nt, 128, -1).max(axis=1)
    return 2.0 ** -50 * 128 * (Xa.T @ Ya) + 4 * nt * 2.0 ** -53 * (np.abs(X).T @ np.abs(Y))


@pytest.mark.parametrize("n,a,b", [(99841, 8, 8), (99855, 11, 5), (99857, 1, 1), (100095, 16, 5), (100001, 3, 13),
                                   (50001, 33, 5), (99841, 1, 20), (99999, 128, 1)])
def test_gram_elementwise(rbo, n, a, b):
    rng = np.random.default_rng(n + 7 * a + b)
    X = rng.standard_normal((n, a)) * 10.0 ** rng.uniform(-8, 8, a)
    Y = rng.standard_normal((n, b)) * 10.0 ** rng.uniform(-8, 8, b)
    ref, bound = ogram(X, Y), _bound(X, Y)
    assert (np.abs(rbo.gram(_dev(rbo, X), _dev(rbo, Y)) - ref) <= bound).all()
    odd = n | 1
    assert (np.abs(rbo.gram(_dev(rbo, X, odd), _dev(rbo, Y, odd)) - ref) <= bound).all()


@pytest.mark.parametrize("n,s,nb,s_hat", [(99841, 5, 4, 0), (99855, 5, 6, 30), (100095, 1, 6, 0), (78001, 8, 4, 16),
                                          (100001, 16, 2, 0), (50015, 10, 3, 30)])
def test_orthogonalization_with_and_without_tensor_copies(rbo, n, s, nb, s_hat):
    """Values over the whole range of a digit (runs of equal bytes) among the Gaussian ones; the
    arithmetic does not depend on how a tile comes in, so the results are equal."""
    V = synth.glued_blocks(n, nb, s, 10.0, seed=n, v0=True)
    V[::7, 0] = np.copysign(0x7F7F7F7F7F7F7F / 2.0 ** 55, V[::7, 0])
    V[3::7, 0] = np.copysign(0x80808080808080 / 2.0 ** 55, V[3::7, 0])
    sk = rbo.sketch_create(n, 4 * (nb * s + 2), 8, 42)
    res = []
    for ld in (n + (n & 1), n | 1):
        D = _dev(rbo, V, ld + 2)
        out = rbo.block_orth_two_stage(sk, D, s, s_hat, v0=True) if s_hat else \
            rbo.block_orth_one_stage(sk, D, s, v0=True)
        res.append((D.cpu().numpy(), out.R))
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
    assert metrics.orth_error(res[0][0]) <= 1e-13
    assert metrics.backward_error(V, *res[0]) <= 1e-14
