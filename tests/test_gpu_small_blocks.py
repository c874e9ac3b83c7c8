"""GPU: every CTA size of the fixed-point FP64 kernel at the edges of its range, on bins that select
it (the selection is read from the plan's log), against the FP64 oracle block by block: one warp a block
up to N = 47, two to eight warps with tiles in shared memory, four or eight with tiles in the
workspace; with two coincident points and with white data, whose rows are scaled during the
factorisation.  And that a block costs what its own size needs, not its tile row's.

Tolerance: tau^2 = 1e-3, N <= 240: a pivot's logarithm errs by at most N 2^-53 (1.3 / 1e-3) < 4e-11 on
either side and the quadratic form by as much relative to itself: 1e-9 absolute plus 1e-9 relative."""
import re
import time

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


@pytest.mark.parametrize("d,nu", [(2, 1.5), (3, 0.5), (2, 1.2)])
@pytest.mark.parametrize("N,blocks,kind,threads", [
    (2, 700, 8, 32), (9, 700, 8, 32), (15, 700, 8, 32), (16, 1400, 8, 32), (17, 1400, 8, 32), (24, 1400, 8, 32),
    (25, 3400, 8, 32), (31, 3400, 8, 32), (16, 700, 7, 64), (25, 1400, 7, 64), (31, 700, 7, 64), (32, 3400, 8, 32), (33, 3400, 8, 32), (40, 3400, 8, 32), (47, 3400, 8, 32),
    (32, 700, 7, 64), (33, 700, 7, 64), (47, 700, 7, 64), (17, 280, 7, 256), (31, 270, 7, 256), (47, 250, 7, 256),
    (48, 700, 8, 128), (64, 700, 8, 128), (111, 700, 8, 128), (112, 700, 9, 128), (239, 400, 9, 128), (240, 400, 9, 256)])
def test_forms(bv, N, blocks, kind, threads, d, nu, monkeypatch, capfd):
    m = N - 1
    n = blocks + m  # blocks of one point in order: the first m have fewer neighbours
    locs = synth.locs_uniform(n, d, 500 + N)
    locs[n - 1] = locs[n - 2]
    y = synth.normal(500 + N, 20, n)
    bp, pi = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32)
    th = (1.3, 0.2, nu, 1e-3)
    monkeypatch.setenv("BV_LOG_PLAN", "1")
    with bv.Context() as ctx:
        ctx.set_data(locs, y)
        ctx.set_blocks(bp, pi, locs)
        nnp, nni = ctx.select_neighbors(m)
        capfd.readouterr()
        ll, per, _ = ctx.loglik(bv.theta(*th), bv.BV_FP64, per_block=True)
        bins = re.findall(r"prec 0 bin nmax (\d+) nwork (\d+) -> kind (\d+) threads (\d+)", capfd.readouterr().err)
        assert ll == ctx.loglik(bv.theta(*th), bv.BV_FP64)
    top = [b for b in bins if int(b[0]) == N]
    assert [(int(b[2]), int(b[3])) for b in top] == [(kind, threads)], bins
    first = n - min(blocks, 250)
    _, ref, _ = oracle.loglik(oracle.theta(*th), locs, y, bp[first:], pi, nnp[first:], nni)
    np.testing.assert_allclose(per[first:], ref, rtol=1e-9, atol=1e-9)
    few = min(m, 40)
    _, ref, _ = oracle.loglik(oracle.theta(*th), locs, y, bp[:few + 1], pi, nnp[:few + 1], nni)
    np.testing.assert_allclose(per[:few], ref, rtol=1e-9, atol=1e-9)


def test_cost_follows_the_size(bv):
    # 40,000 blocks: N = 8 against 15 is half of the pivots (and of the covariance), N = 18 against 31 one
    # panel of 16 and two columns against two panels; with whole tile rows each pair took equal times
    import torch
    n = 40_000
    locs = synth.locs_uniform(n, 2, 6)
    best = {}
    for N in (8, 15, 18, 31):
        with bv.Context() as ctx:
            ctx.set_data(locs, synth.normal(6, 20, n))
            ctx.build_singletons(seed=6)
            ctx.select_neighbors(N - 1)
            th = bv.theta(1.0, 0.1, 0.5, 1.0)
            ctx.loglik(th, bv.BV_FP64)
            ts = []
            for _ in range(12):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                ctx.loglik(th, bv.BV_FP64)
                ts.append(time.perf_counter() - t0)
            best[N] = min(ts)
    assert best[8] <= 0.9 * best[15] and best[18] <= 0.9 * best[31], best
