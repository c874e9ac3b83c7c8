"""GPU: K-means blocks of several threads at a time, each with its own context and number of
dimensions (the one-launch seeding's shared memory grows with it): every call succeeds with the blocks
that it gives alone."""
import threading

import numpy as np
import pytest

from paper_2410_04477_gb300 import synth

pytestmark = pytest.mark.gpu


def test_kmeans_of_several_dimensions_at_once():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_04477_gb300 import bv
    sets = {d: synth.locs_uniform(40_000, d, 31 + d) for d in (1, 2, 3)}

    def blocks(d):
        with bv.Context() as ctx:
            ctx.set_data(sets[d])
            return ctx.build_blocks(8, seed=3, iters=1)

    want = {d: blocks(d) for d in sets}
    errors = []

    def work(d):
        try:
            for _ in range(25):
                bp, pi = blocks(d)
                assert np.array_equal(bp, want[d][0]) and np.array_equal(pi, want[d][1])
        except Exception as e:  # (an assertion of a thread would be lost)
            errors.append((d, repr(e)))

    threads = [threading.Thread(target=work, args=(d,)) for d in (1, 2, 3, 3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
