"""GPU: distances at the ends of FP64's range: squares that overflow, and the smallest whose squares are
normal numbers."""
import numpy as np
import pytest

import oracle
from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [0.5, 0.8, 1.5])
def test_overflowing_distances(nu):
    # the exact likelihood takes them as a covariance of 0 where the form has that limit (nu = 1/2, K_nu), as
    # a merely large distance; the polynomial forms are refused, and the block likelihood refuses all
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv
    n = 24
    near = synth.locs_uniform(n, 2, 3)
    far = near.copy()
    near[-2:] = [[1e4, 0.0], [0.0, -1e4]]          # 1e5 ranges away: the covariance underflows
    far[-2:] = [[1e200, 0.0], [0.0, -3e201]]
    y = synth.normal(3, 20, n)
    th = (1.0, 0.1, nu, 1e-2)
    with bv.Context() as ctx:
        ctx.set_data(far, y)
        ctx.set_blocks(np.array([0, n], np.int64), np.arange(n, dtype=np.int32), far[:1].copy())
        ctx.select_neighbors(0)
        with pytest.raises(bv.BVError):
            ctx.loglik(bv.theta(*th), bv.BV_FP64)
        if nu == 1.5:
            with pytest.raises(bv.BVError):
                ctx.exact_loglik(bv.theta(*th))
        else:
            want = oracle.exact_loglik(oracle.theta(*th), near, y)
            assert abs(ctx.exact_loglik(bv.theta(*th))[0] - want) <= 1e-10 * abs(want)


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
