"""The pivots' own step of the fixed-point factorisation, a - x^2: the function on the CPU against
whole numbers, and on the GPU the second pivot of pairs of points at close distances, which is
1 - e^(-2 x) without a nugget."""
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_04477_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "bv_fix.cuh"
int main() {
    long long a, x;
    while (scanf("%lld %lld", &a, &x) == 2)
        printf("%lld\n", (long long)bvfix::sub_square(a, x, (int32_t)((x + (1ll << 28)) >> 29)));
}
"""


def test_square_is_rounded_once(tmp_path):
    # half a unit of the rounding and l l's cut to 14 bits (2 l 2^15 2^-58 < 2^-13)
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rng = np.random.default_rng(5)
    xs = [0, 1, -1, 1 << 59, -(1 << 59), (1 << 59) - 1, (1 << 28), (1 << 28) - 1, (1 << 59) - (1 << 28), 3 << 57]
    xs += [int(v) for v in rng.integers(-(1 << 59), 1 << 59, 4000)] + [int(v) >> int(s) for v, s in zip(rng.integers(1 << 58, 1 << 59, 500), rng.integers(0, 59, 500))]
    cases = [(1 << 60, x) for x in xs]
    out = subprocess.run([str(exe)], input="\n".join(f"{a} {x}" for a, x in cases), capture_output=True, text=True)
    got = [int(v) for v in out.stdout.split()]
    assert len(got) == len(cases)
    for (a, x), v in zip(cases, got):
        assert abs((v - a) * (1 << 58) + x * x) <= (1 << 57) + (1 << 45), (x, v)


@pytest.mark.gpu
def test_pivot_of_close_pairs():
    # entry: z's rounding (2.8 units of 2^-60) and two products, 4 units, twice in the pivot; the
    # solved entry's rounding (half a unit of 2^-59), 2 units; the step's own half: below 16 units.
    # Scaled distances j 2^-26 and their squares are exact
    from paper_2410_04477_gb300 import bv
    j = np.concatenate([np.arange(1, 40), np.arange(40, 4000, 97)])
    k = len(j)
    locs = np.zeros((2 * k, 2))
    locs[0::2, 0] = np.arange(k) / 64.0
    locs[1::2, 0] = locs[0::2, 0] + j * 2.0 ** -27
    x = j * 2.0 ** -26
    p2 = -np.expm1(-2.0 * x)
    want = -0.5 * (np.log(p2) + 2.0 * math.log(2.0 * math.pi))
    with bv.Context() as ctx:
        ctx.set_data(locs, np.zeros(2 * k))
        ctx.set_blocks(2 * np.arange(k + 1, dtype=np.int64), np.arange(2 * k, dtype=np.int32), locs[0::2].copy())
        ctx.select_neighbors(0)
        _, per, _ = ctx.loglik(bv.theta(1.0, 0.5, 0.5, 0.0), bv.BV_FP64, per_block=True)
    assert np.all(np.abs(per - want) <= 0.5 * 16 * 2.0 ** -60 / p2 + 2e-14), np.max(np.abs(per - want) * 2 * p2) * 2.0 ** 60
