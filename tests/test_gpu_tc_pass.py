"""Row passes on the tensor cores (exact fixed-point digits) at the sizes where they can go
wrong: tile and fragment edges, unaligned arrays (plain loads), groups that fall back to
float64, scales that change between tiles, and both forms of the sketched panel step.

Bound of the digit Gram, per chunk of at most 64 rows with largest magnitudes Mx, My: a
value is off by less than 2^-54 of its column's largest, and the digit pairs left out weigh
less than 2^-53.4 Mx My per row, so a chunk is off by at most 64 Mx My (2^-53 + 2^-53.4);
joining a chunk and adding it to the float64 sum round once each, at most
2 (chunks) 2^-53 of |X|^T |Y|, and the reduction over CTAs adds at most 2^-53 |X|^T |Y| per
CTA.  The test allows 2^-51 sum_chunks 64 Mx My + (4 chunks) 2^-53 |X|^T |Y|."""
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
    nt = (n + 63) // 64
    pad = ((0, nt * 64 - n), (0, 0))
    Xa = np.abs(np.pad(X, pad)).reshape(nt, 64, -1).max(axis=1)
    Ya = np.abs(np.pad(Y, pad)).reshape(nt, 64, -1).max(axis=1)
    return 2.0 ** -51 * 64 * (Xa.T @ Ya) + 4 * nt * 2.0 ** -53 * (np.abs(X).T @ np.abs(Y))


@pytest.mark.parametrize("odd_ld", [False, True])
@pytest.mark.parametrize("n,a,b", [(1, 1, 1), (15, 3, 2), (16, 16, 8), (17, 17, 9), (63, 8, 8), (64, 33, 5),
                                   (65, 40, 7), (129, 48, 16), (1000, 64, 5), (4099, 128, 3), (777, 65, 30),
                                   (30011, 15, 5), (257, 1, 64)])
def test_gram_elementwise(rbo, n, a, b, odd_ld):
    rng = np.random.default_rng(n + 7 * a + b)
    X = rng.standard_normal((n, a)) * 10.0 ** rng.uniform(-8, 8, a)
    Y = rng.standard_normal((n, b)) * 10.0 ** rng.uniform(-8, 8, b)
    X[: n // 2, 0] *= 1e-10
    Y[:, b - 1] *= np.where(np.arange(n) % 3 == 0, 1.0, 2.0 ** -30)  # widely graded inside a chunk
    if a > 2:
        X[:, 1] = 0.0
        X[n // 3, 2] = 1e12
    ld = n + 1 - (n & 1) if odd_ld else None
    C = rbo.gram(_dev(rbo, X, ld), _dev(rbo, Y, ld))
    assert (np.abs(C - ogram(X, Y)) <= _bound(X, Y)).all()


def test_gram_groups_outside_the_fixed_point_range(rbo):
    n = 1000
    rng = np.random.default_rng(5)
    X = rng.standard_normal((n, 9))
    Y = rng.standard_normal((n, 4))
    X[:, 0] *= 1e-300
    X[:, 1] *= 1e300
    X[:, 2] = 0.0
    X[:, 3] = 5e-320          # a subnormal column
    Y[:, 1] *= 1e-200
    Y[:, 2] *= 1e8
    X[501:, 4] *= 1e-290      # changes range between chunks
    C = rbo.gram(_dev(rbo, X), _dev(rbo, Y))
    # float64 products and sums of n terms in any order, and results that underflow; an
    # entry whose terms overflow float64 (1e300 by 1e8) has no bound
    with np.errstate(over="ignore"):
        ref = ogram(X, Y)
        tol = n * 2.0 ** -52 * (np.abs(X).T @ np.abs(Y)) + 1e-322
    fits = np.isfinite(tol)
    assert fits.sum() == fits.size - 1
    assert (np.abs(C - ref)[fits] <= tol[fits]).all()
    X[7, 5], X[900, 6], Y[3, 0] = np.nan, np.inf, -np.inf
    C = rbo.gram(_dev(rbo, X), _dev(rbo, Y))
    bad = np.zeros(fits.shape, dtype=bool)
    bad[5], bad[6], bad[:, 0] = True, True, True
    assert not np.isfinite(C[bad]).any()
    good = fits & ~bad
    assert (np.abs(C - ref)[good] <= tol[good]).all()


@pytest.mark.parametrize("n,s,nb", [(65, 5, 3), (1001, 4, 9), (4097, 8, 5), (333, 16, 4), (2000, 7, 7)])
@pytest.mark.parametrize("s_hat", [0, 1])
def test_unaligned_columns_match_aligned(rbo, n, s, nb, s_hat):
    """Odd leading dimension (plain loads, scalar write-back) against the tensor copies: the
    same arithmetic in the same order, so the results are equal."""
    V = synth.glued_blocks(n, nb, s, 10.0, seed=n, v0=True)
    sk = rbo.sketch_create(n, 4 * (nb * s + 2), 8, 42)
    out = []
    for ld in (n + (n & 1), n + 1 - (n & 1)):
        D = _dev(rbo, V, ld)
        if s_hat:
            r = rbo.block_orth_two_stage(sk, D, s, s * nb if s * nb <= 64 else s, v0=True)
        else:
            r = rbo.block_orth_one_stage(sk, D, s, v0=True)
        out.append((D.cpu().numpy(), r.R))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    Q, R = out[0]
    assert metrics.orth_error(Q) <= 1e-13 and metrics.backward_error(V, Q, R) <= 1e-14


@pytest.mark.parametrize("n,k,d,zeta", [(1, 1, 16, 1), (63, 5, 244, 8), (64, 8, 40, 8), (70001, 5, 244, 8),
                                        (5000, 16, 300, 4), (4099, 10, 404, 16), (2000, 3, 4096, 8)])
def test_sketch_sums_with_growing_scale(rbo, n, k, d, zeta):
    """Every value is rounded at 2^-53 of its column's largest so far, the tile sums are
    exact, and the float64 partials are added once per 512 rows and CTA; shifting the sums
    when the scale grows rounds at the same unit (at most 2048 shifts)."""
    rng = np.random.default_rng(n)
    W = rng.standard_normal((n, k)) * 10.0 ** rng.uniform(-8, 8, k)
    W *= (2.0 ** (np.arange(n) * 60.0 / n - 60.0))[:, None]  # grows by 2^60 over the rows
    sk = rbo.sketch_create(n, d, zeta, 42)
    got = rbo.sketch_apply(sk, _dev(rbo, W))
    idx, sg = (t.cpu().numpy() for t in rbo.sketch_entries(sk, 0, n))
    ref, cnt = np.zeros((d, k), dtype=np.longdouble), np.zeros(d)
    for j in range(zeta):
        np.add.at(ref, idx[:, j], sg[:, j][:, None] * W.astype(np.longdouble))
        np.add.at(cnt, idx[:, j], 1.0)
    bound = (2 * cnt + 64.0)[:, None] * 2.0 ** -52 * np.abs(W).max(axis=0)[None, :]
    assert (np.abs(got - ref) <= bound).all()
    W[n // 2, 0] = np.nan
    assert np.isnan(rbo.sketch_apply(sk, _dev(rbo, W))[:, 0]).all()


@pytest.mark.parametrize("s,s_hat,d", [(1, 6, 64), (3, 9, 40), (16, 48, 200), (16, 16, 16), (20, 40, 170), (5, 60, 61)])
def test_two_stage_panel_widths(rbo, s, s_hat, d):
    """Panels of at most 16 columns run the sketched BCGS2-HH on a cluster, wider ones in the
    last CTA of the pass: R of a well-conditioned V is the Householder R to rounding."""
    n = 3001
    V = synth.glued_blocks(n, s_hat // s, s, 10.0, seed=s, v0=True) if s > 1 else \
        np.random.default_rng(1).standard_normal((n, s_hat + 1))
    sk = rbo.sketch_create(n, d, 8, 42)
    D = _dev(rbo, V)
    out = rbo.block_orth_two_stage(sk, D, s, s_hat, v0=True)
    R = np.linalg.qr(V, mode="r")
    R *= np.sign(np.diag(R))[:, None]
    assert metrics.rel_diff(out.R, R) <= 1e-12
    assert metrics.orth_error(D.cpu().numpy()) <= 1e-13
