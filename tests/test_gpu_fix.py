"""GPU: the fixed-point FP64 kernel against the FP64 oracle, block by block, at the sizes
where it can go wrong: N just below, at and above multiples of its 16-row tiles (the data
row then ends a tile, or has one to itself), the switches of CTA size and of where the
tiles live, and the largest N; closed-form and general smoothness, 1 to 3 dimensions,
coincident and nearly coincident points, and data rows that leave the fixed-point range.

Tolerance: a pivot's error is at most about N 2^-53 of sigma^2 + tau^2 on either side, so its
logarithm errs by N 2^-53 (sigma^2 + tau^2) / tau^2 < 1e-10 for N <= 400, tau^2 >= 1e-3, and
the quadratic form by that times itself: 1e-9 absolute plus 1e-9 relative."""
import numpy as np
import pytest

import oracle
from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bv():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv as _bv
    return _bv


def _compare(bv, locs, y, bp, pi, cen, m, th, ranges=None, rtol=1e-9, atol=1e-9):
    with bv.Context() as ctx:
        ctx.set_data(locs, y)
        ctx.set_blocks(bp, pi, cen)
        nnp, nni = ctx.select_neighbors(m)
        ll, per, _ = ctx.loglik(bv.theta(*th, ranges=ranges), bv.BV_FP64, per_block=True)
        again = ctx.loglik(bv.theta(*th, ranges=ranges), bv.BV_FP64)
    ref, per_ref, _ = oracle.loglik(oracle.theta(*th, ranges=ranges), locs, y, bp, pi, nnp, nni)
    np.testing.assert_allclose(per, per_ref, rtol=rtol, atol=atol)
    assert ll == again
    return np.diff(bp) + np.diff(nnp)


def _blocks(n, sizes):
    bp = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    assert bp[-1] == n
    return bp, np.arange(n, dtype=np.int32)


@pytest.mark.parametrize("N", [2, 14, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 79, 80, 111, 112, 113, 128, 175, 239, 240, 300])
@pytest.mark.parametrize("form", [(2, 1.5), (3, 0.5), (1, 2.5), (2, 1.2)])
def test_tile_edges(bv, N, form):
    d, nu = form
    b = 3 if N > 4 else 1
    m, n = N - b, N + 9 * b
    locs = synth.locs_uniform(n, d, 300 + N)
    sizes = [b] * (n // b) + ([n % b] if n % b else [])
    bp, pi = _blocks(n, sizes)
    cen = np.add.reduceat(locs, bp[:-1], axis=0) / np.diff(bp)[:, None]
    th = (1.3, 0.2, nu, 1e-3 if nu != 2.5 else 1e-2)
    y = oracle.exact_draw(oracle.theta(*th), locs, synth.normal(300 + N, 20, n))
    Ns = _compare(bv, locs, y, bp, pi, cen, m, th)
    assert Ns.max() == N


def test_largest_shared_size_and_beyond(bv):
    # one block of all points: the panel's rows need more than one pass (N = 600), and a block
    # too large for the kernel goes to the global-memory one (N = 1500)
    for n in (600, 1500):
        locs = synth.locs_uniform(n, 2, 77 + n)
        th = (1.0, 0.1, 0.5, 1e-2)
        y = oracle.exact_draw(oracle.theta(*th), locs, synth.normal(77, 20, n))
        bp, pi = _blocks(n, [n])
        _compare(bv, locs, y, bp, pi, locs.mean(axis=0, keepdims=True), 0, th)


@pytest.mark.parametrize("nu", [0.5, 1.5, 2.5, 0.35, 3.1])
def test_coincident_and_near_points(bv, nu):
    # distances 0, 1e-14, 1e-9 and 1e-5 ranges: below the table of the general smoothness, and
    # within it; far pairs (500 ranges) whose covariance is 0
    n = 90
    locs = synth.locs_uniform(n, 2, 411) * 30.0
    locs[1], locs[2], locs[3], locs[4] = locs[0], locs[0] + 1e-15, locs[0] + [0.0, 1e-10], locs[0] + [1e-6, 0.0]
    th = (0.7, 0.06, nu, 1e-2)
    y = synth.normal(411, 20, n)
    bp, pi = _blocks(n, [30, 30, 30])
    cen = np.add.reduceat(locs, bp[:-1], axis=0) / 30.0
    _compare(bv, locs, y, bp, pi, cen, 40, th)


@pytest.mark.parametrize("scale", [1.0, 1e-9, 1e12])
def test_data_row_out_of_range(bv, scale):
    # white data under a smooth covariance with a small nugget: conditional standardised values
    # near 1 / sqrt(tau^2) = 300, far beyond the data row's headroom of 2^5, so blocks are done
    # again at a wider scale; tau^2 = 1e-5 brings the pivots' relative error to about N 2^-53 1e5
    n = 400
    locs = synth.locs_uniform(n, 2, 512)
    th = (1.0, 0.4, 2.5, 1e-5)
    y = scale * synth.normal(512, 20, n)
    bp, pi = _blocks(n, [10] * 40)
    cen = np.add.reduceat(locs, bp[:-1], axis=0) / 10.0
    _compare(bv, locs, y, bp, pi, cen, 60, th, rtol=1e-8, atol=1e-8)


def test_extreme_scales(bv):
    # the covariance is normalised by its diagonal: a tiny and a huge sigma^2
    n = 300
    locs = synth.locs_uniform(n, 2, 613)
    z = synth.normal(613, 20, n)
    bp, pi = _blocks(n, [10] * 30)
    cen = np.add.reduceat(locs, bp[:-1], axis=0) / 10.0
    for s2 in (1e-200, 1e200):
        th = (s2, 0.1, 1.5, 1e-2 * s2)
        _compare(bv, locs, np.sqrt(s2) * z, bp, pi, cen, 45, th)


@pytest.mark.parametrize("n", [15, 16, 17, 64, 79, 80, 128, 129, 257, 700])
def test_exact_tile_edges(bv, n):
    # the dense factorisation at the edges of its 16-row tiles and 64-column panels, and with a
    # data row that has to be rescaled (white data: standardised values near 1 / sqrt(tau^2));
    # tau^2 = 1e-4: pivots within n 2^-53 1e4, 1e-9 of their logarithms' sum
    locs = synth.locs_uniform(n, 2, 700 + n)
    y = synth.normal(700 + n, 20, n)
    for nu in (1.5, 0.8):
        th = (1.1, 0.3, nu, 1e-4)
        with bv.Context() as ctx:
            ctx.set_data(locs, y)
            ll, quad, ld = ctx.exact_loglik(bv.theta(*th))
        want = oracle.exact_loglik(oracle.theta(*th), locs, y)
        assert abs(ll - want) <= 1e-9 * max(1.0, abs(want), quad), (nu, ll, want)


@pytest.mark.parametrize("m", [1, 15, 16, 17, 47, 64, 120, 200])
@pytest.mark.parametrize("nu", [0.5, 2.5, 0.9])
def test_prediction_tile_edges(bv, m, nu):
    # the partial elimination with m below, at and above whole panels of 16; white data under a
    # smooth covariance, so that the data row is rescaled; tau^2 = 1e-3: errors of about
    # N 2^-53 1e3 of the prior's scale and of the data's
    n, ns = 500, 60
    locs, star = synth.locs_uniform(n, 2, 800), synth.locs_uniform(ns, 2, 801)
    y = synth.normal(800, 20, n)
    th = (1.0, 0.25, nu, 1e-3)
    with bv.Context() as ctx:
        ctx.set_data(locs, y)
        ctx.set_pred_locations(star)
        bp, pi = ctx.build_pred_blocks(6, seed=3)
        nnp, nni = ctx.select_pred_neighbors(m)
        mean, var, cov = ctx.predict(bv.theta(*th), packed_cov=True)
    omean, ovar, ocov = oracle.predict(oracle.theta(*th), locs, y, star, bp, pi, nnp, nni, packed_cov=True)
    np.testing.assert_allclose(mean, omean, rtol=1e-9, atol=1e-9)
    np.testing.assert_allclose(var, ovar, rtol=1e-9, atol=1e-11)
    np.testing.assert_allclose(cov, ocov, rtol=1e-9, atol=1e-11)


@pytest.mark.parametrize("n,k,d", [(8192, 40, 2), (8193, 40, 3), (20000, 64, 1), (40960, 24, 2), (40961, 24, 2), (300, 300, 2)])
def test_kmeans_seeding_forms(bv, n, k, d):
    # one to five points a thread of the one-launch seeding, its largest set and the first one
    # beyond, every point a centre, and repeated points (weights of zero): the oracle's blocks
    locs = synth.locs_uniform(n, d, 900 + d)
    locs[n // 2:n // 2 + 40] = locs[:40]
    with bv.Context() as ctx:
        ctx.set_data(locs)
        bp, pi = ctx.build_blocks(k, seed=11, iters=2)
    obp, opi, _ = oracle.build_blocks(locs, k, seed=11, iters=2)
    np.testing.assert_array_equal(bp, obp)
    np.testing.assert_array_equal(pi, opi)
