"""sigma^2 / D, which scales every covariance entry of the fixed-point kernels, to 63 bits: the
function itself on the CPU (all sizes of both numbers) against whole-number division, and on the
GPU the pivot of two coincident points with a small nugget, which it alone decides."""
import math
import os
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_04477_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "bv_fix.cuh"
int main() {
    double a, b;
    while (scanf("%la %la", &a, &b) == 2) printf("%llu\n", (unsigned long long)bvfix::ratio63(a, b));
}
"""


def test_ratio_is_rounded_to_63_bits(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rng = np.random.default_rng(3)
    pairs = [(1.0, 1.0), (1.0, 1.0001), (1.0, 1.001), (1.0, 1.0 + 1e-6), (5e-324, 5e-324), (5e-324, 1e308), (1e308, 1.7e308),
             (1.0, 2.0 ** 63), (1.0, 2.0 ** 64), (1.0, 2.0 ** 65), (1.5, 2.0 ** 65), (1.0, 3.0 * 2.0 ** 62)]
    for _ in range(3000):
        s = float(np.exp(rng.uniform(-40, 40)))
        pairs.append((s, s + s * float(np.exp(rng.uniform(-45, 50)))))
    out = subprocess.run([str(exe)], input="\n".join(f"{a.hex()} {b.hex()}" for a, b in pairs), capture_output=True, text=True)
    got = [int(v) for v in out.stdout.split()]
    assert len(got) == len(pairs)
    for (a, b), v in zip(pairs, got):
        assert abs(v - F(a) / F(b) * 2 ** 63) <= F(1, 2), (a, b, v)


@pytest.mark.gpu
@pytest.mark.parametrize("tau2", [1e-9, 3e-9, 7e-9, 1.1e-8])
@pytest.mark.parametrize("sigma2", [1.0, 0.7])
def test_pivot_of_coincident_points(tau2, sigma2):
    # two points in one place: the second pivot is 1 - (sigma^2 / D)^2 = 2 tau^2, of which one unit
    # of 2^-60 in sigma^2 / D is two.  The entry is within 2 units (a product and a shift), the
    # pivot's own step within 2 more: 8 units of 2^-60 in all, doubled
    from paper_2410_04477_gb300 import bv
    locs = np.array([[0.25, 0.5], [0.25, 0.5]])
    D = sigma2 + tau2
    det = F(D) ** 2 - F(sigma2) ** 2
    p2 = det / F(D)                                     # the second pivot
    want = -0.5 * (math.log(D) + math.log(p2) + 2.0 * math.log(2.0 * math.pi))
    tol = 0.5 * 16 * 2.0 ** -60 / float(p2 / F(D)) + 2e-14
    with bv.Context() as ctx:
        ctx.set_data(locs, np.zeros(2))
        ctx.set_blocks(np.array([0, 2], np.int64), np.array([0, 1], np.int32), locs[:1].copy())
        ctx.select_neighbors(0)
        for nu in (0.5, 1.5, 2.5, 0.8):
            ell = ctx.loglik(bv.theta(sigma2, 0.1, nu, tau2), bv.BV_FP64)
            assert abs(ell - want) <= tol, (nu, ell, want)
            ell = ctx.exact_loglik(bv.theta(sigma2, 0.1, nu, tau2))[0]
            assert abs(ell - want) <= tol, (nu, ell, want)
    # prediction there: the conditional variance is that pivot (with 39 far sites in the block, so that it
    # takes the fixed-point kernel)
    with bv.Context() as ctx:
        ctx.set_data(locs[:1], np.zeros(1))
        ctx.set_pred_locations(np.concatenate([locs[:1], locs[:1] + 100.0 * np.arange(1, 40)[:, None]]))
        ctx.build_pred_blocks(1, seed=1)
        ctx.select_pred_neighbors(1)
        for nu in (0.5, 1.5, 2.5, 0.8):
            var = ctx.predict(bv.theta(sigma2, 0.1, nu, tau2))[1]
            assert abs(var[0] - float(p2)) <= 16 * 2.0 ** -60 * D + 1e-15 * float(p2), (nu, var[0], float(p2))
