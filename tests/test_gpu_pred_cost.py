"""GPU: what prediction costs follows the sizes of its blocks: with a general smoothness the pairs of
points (each a K_nu), not whole tiles; with a closed form, small blocks do not pay for the panels of larger
ones."""
import time

import numpy as np
import pytest

from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


def _times(cases, n_star, blocks):
    """Least time of a prediction per case (m, theta), the context's set-up apart."""
    import torch
    from paper_2410_04477_gb300 import bv
    locs, star = synth.locs_uniform(8000, 2, 1), synth.locs_uniform(n_star, 2, 2)
    y = synth.normal(1, 20, 8000)
    best = {}
    for m, th in cases:
        with bv.Context() as ctx:
            ctx.set_data(locs, y)
            ctx.set_pred_locations(star)
            ctx.build_pred_blocks(blocks, seed=1, iters=1)
            ctx.select_pred_neighbors(m)
            t = bv.theta(*th)
            ctx.predict(t)
            ts = []
            for _ in range(6):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                ctx.predict(t)
                ts.append(time.perf_counter() - t0)
            best[m] = min(ts)
    return best


def test_general_smoothness_costs_its_pairs():
    # m = 33 and 47 fill the same tiles; 561 against 1,128 pairs of points
    th = (1.0, 0.05, 0.8, 1e-2)
    best = _times([(33, th), (47, th)], 4000, 4000)
    assert best[33] <= 0.8 * best[47], best


def test_small_blocks():
    # 2 neighbours against 31 at 20,000 single sites: 6 entries against 528, and a thousandth of the
    # operations; at least three times as fast (in whole panels of the fixed-point kernel: 1.8)
    th = (1.0, 0.05, 1.5, 1e-2)
    best = _times([(2, th), (31, th)], 20_000, 20_000)
    assert 3.0 * best[2] <= best[31], best


@pytest.mark.parametrize("m", [21, 22, 23])
def test_both_kernels_at_their_limit(m):
    # blocks of 10 sites: 31, 32 and 33 points a block, where the FP64 kernel hands over to the fixed-point
    # one; tau^2 = 1e-2: errors of N 2^-53 1e2 < 1e-12 of the prior's and the data's scale
    import oracle
    from paper_2410_04477_gb300 import bv
    locs, star = synth.locs_uniform(600, 2, 5), synth.locs_uniform(400, 2, 6)
    y = synth.normal(5, 20, 600)
    with bv.Context() as ctx:
        ctx.set_data(locs, y)
        ctx.set_pred_locations(star)
        bp, pi = ctx.build_pred_blocks(40, seed=3)
        nnp, nni = ctx.select_pred_neighbors(m)
        for nu in (0.5, 1.5, 2.5, 0.8):
            th = (1.2, 0.2, nu, 1e-2)
            mean, var, cov = ctx.predict(bv.theta(*th), packed_cov=True)
            om, ov, oc = oracle.predict(oracle.theta(*th), locs, y, star, bp, pi, nnp, nni, packed_cov=True)
            np.testing.assert_allclose(mean, om, rtol=1e-10, atol=1e-10)
            np.testing.assert_allclose(var, ov, rtol=1e-10)
            np.testing.assert_allclose(cov, oc, rtol=1e-10, atol=1e-11)
