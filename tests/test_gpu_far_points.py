"""GPU: points whose scaled squared distance leaves FP64's range: at nu = 1/2 their covariance is 0, in
the block likelihood, the exact one and in prediction, as with a merely large distance."""
import numpy as np
import pytest

import oracle
from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


def test_overflowing_distances():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv
    n = 24
    locs = synth.locs_uniform(n, 2, 3)
    near, far = locs.copy(), locs.copy()
    near[-2:] = [[1e4, 0.0], [0.0, -1e4]]          # 1e5 ranges away: the covariance underflows
    far[-2:] = [[1e200, 0.0], [0.0, -3e201]]       # the squared distance overflows
    y = synth.normal(3, 20, n)
    th = (1.0, 0.1, 0.5, 1e-2)
    got = []
    for pts in (near, far):
        with bv.Context() as ctx:
            ctx.set_data(pts, y)
            ctx.set_blocks(np.array([0, n], np.int64), np.arange(n, dtype=np.int32), locs[:1].copy())
            ctx.select_neighbors(0)
            got.append((ctx.loglik(bv.theta(*th), bv.BV_FP64), ctx.exact_loglik(bv.theta(*th))[0]))
    want = oracle.exact_loglik(oracle.theta(*th), near, y)
    assert got[0] == got[1]
    np.testing.assert_allclose(got[0], want, rtol=1e-10)
    # prediction at a far point from all observations: the prior
    with bv.Context() as ctx:
        ctx.set_data(locs[:20], y[:20])
        ctx.set_pred_locations(far[-2:])
        ctx.build_pred_blocks(1, seed=1)
        ctx.select_pred_neighbors(20)
        mean, var, _ = ctx.predict(bv.theta(*th))
    np.testing.assert_allclose(mean, 0.0, atol=1e-12)
    np.testing.assert_allclose(var, 1.01, rtol=1e-14)


@pytest.mark.parametrize("x", [2.0 ** -499.5, 2.0 ** -503.5, 2.0 ** -508.5])
def test_distances_near_the_smallest(x):
    # a general smoothness near 0 still tells 2^-510 ranges (the smallest whose square is a normal number)
    # from 0: 1 - rho of about x^(2 nu) / 2; the covariance within 1e-13 (log rho = nu log x + log K_nu,
    # |log K_nu| < 10, in FP64), the pivot above tau^2 = 1e-2: 1e-10
    from paper_2410_04477_gb300 import bv
    n = 12
    locs = synth.locs_uniform(n, 1, 4)
    locs[0], locs[1] = 0.0, x
    y = synth.normal(4, 20, n)
    th = (1.0, 1.0, 0.02, 1e-2)
    bp, pi = np.array([0, n], np.int64), np.arange(n, dtype=np.int32)
    with bv.Context() as ctx:
        ctx.set_data(locs, y)
        ctx.set_blocks(bp, pi, locs[:1].copy())
        nnp, nni = ctx.select_neighbors(0)
        ell = ctx.loglik(bv.theta(*th), bv.BV_FP64)
    want, _, _ = oracle.loglik(oracle.theta(*th), locs, y, bp, pi, nnp, nni)
    assert abs(ell - want) <= 1e-10 * max(1.0, abs(want)), (ell, want)
