"""GPU: the rounding of conditional simulation's sample mean with few rounds, against extended precision.

Prior sites (observations of 0 far away): every draw is sd z.  With R = 2 the middle of the interval
is sd (z_0 + z_1) / 2, of size 0.7.  Its RMS error: the interval's ends, their mean and sd zbar are rounded
once each (values of 0.3 to 1: 2^-54.8 each on average, the two ends 2^-55.3 together), the pair's
sum to 2^-54 (2^-55.8, halved): 2^-53.9 in all; limit 2^-53.4.  (Draws rounded to 2^-50: 2^-52.6.)"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _draws(seed, n, rounds, first):
    """z_0 .. of every location in extended precision, by the stated stream and pair rule."""
    stream = seed ^ 0x636F6E6473696D5F
    half = (rounds + 1) // 2
    L = np.longdouble
    z = np.zeros((n, 2 * half), L)
    two_pi = 2 * L("3.14159265358979323846264338327950288419716939937510")
    for j in range(n):
        for k in range(half):
            c = j * half + k
            u1 = L(1) - L(oracle.splitmix64(stream, 2 * c) >> 11) * L(2) ** -53
            u2 = L(oracle.splitmix64(stream, 2 * c + 1) >> 11) * L(2) ** -53
            rho = np.sqrt(-2 * np.log(u1))
            z[j, 2 * k], z[j, 2 * k + 1] = rho * np.cos(two_pi * u2), rho * np.sin(two_pi * u2)
    return z[:, :rounds]


def test_mean_of_two_draws():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv
    n = 3000
    star = np.column_stack([np.arange(n) * 10.0, np.zeros(n)])
    with bv.Context() as ctx:
        ctx.set_data(np.array([[0.0, 1e6], [1.0, 1e6]]), np.zeros(2))
        ctx.set_pred_locations(star)
        ctx.build_pred_blocks(n, seed=1)
        ctx.select_pred_neighbors(1)
        mean, var, _ = ctx.predict(bv.theta(1.0, 0.1, 0.5, 1e-2))
        lo, up, _ = ctx.cond_sim(rounds=2, seed=77, z_crit=1e-3)
    assert np.all(mean == 0.0) and np.all(var == 1.01)
    z = _draws(77, n, 2, 0)
    want = np.sqrt(np.longdouble(1.01)) * z.mean(axis=1)
    err = (lo.astype(np.longdouble) + up.astype(np.longdouble)) / 2 - want
    assert float(np.sqrt(np.mean(err * err))) <= 2.0 ** -53.4, float(np.sqrt(np.mean(err * err))) * 2.0 ** 53
