"""GPU: what prediction costs follows the sizes of its blocks: with a general smoothness the pairs of
points (each a K_nu), not whole tiles."""
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
