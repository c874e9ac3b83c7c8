"""GPU: k-means++ seeding where the one-launch form's cluster cannot be placed: the form with two
launches a pick takes its place, with the oracle's blocks."""
import time

import numpy as np
import pytest

import oracle
from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


def test_seeding_without_a_cluster(monkeypatch):
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv
    n, k = 9000, 700
    locs = synth.locs_uniform(n, 2, 17)
    seen, cost = [], []
    for fault in ("0", "1"):
        monkeypatch.setenv("BV_FAULT_CLUSTER", fault)
        with bv.Context() as ctx:
            ctx.set_data(locs)
            ctx.build_blocks(k, seed=5, iters=0)
            t0 = time.perf_counter()
            seen.append(ctx.build_blocks(k, seed=5, iters=0))
            cost.append(time.perf_counter() - t0)
    obp, opi, _ = oracle.build_blocks(locs, k, seed=5, iters=0)
    for bp, pi in seen:
        np.testing.assert_array_equal(bp, obp)
        np.testing.assert_array_equal(pi, opi)
    # two launches a pick take at least 5 us, the one-launch form's exchange less than 4.5: the two differ,
    # so the second run did take the other form
    assert cost[1] > 1.5 * cost[0], cost
