"""The fixed-point arithmetic of the FP64 block kernel (csrc/bv_fix.cuh), built for the host:
reciprocal square root, scaled distance, the Matern correlations and the simulation's
Box-Muller pairs against extended precision.  Bounds: the kernel needs correlations within 2^-54 of 1 (the FP64 rounding of a
value near 1); by its steps the square root is within 2^-58 relative and the correlation
within 2^-55 (2^-57 from z's last bit, the rest from five truncated products)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_04477_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "bv_fix.cuh"
using namespace bvfix;
typedef long double L;
static uint64_t A[256], B[256];
static L corr(int nu, L x) { return expl(-x) * (nu == 0 ? 1 : nu == 1 ? 1 + x : 1 + x + x * x / 3); }
int main() {
    std::mt19937_64 g(7);
    L er = 0, ed = 0, ec[3] = {0, 0, 0};
    for (int i = 0; i < 300000; ++i) {
        int64_t p = i < 61 ? 1ll << i : (int64_t)(((g() >> 4) | 1ull << 59) >> (g() % 60));
        if (p < 1) p = 1;
        const Rsq o = rsqrt_fix(p);
        const L t = 1 / sqrtl((L)p * 0x1p-60L), v = ldexpl((L)o.r, o.e - 62);
        er = fmaxl(er, fabsl(v / t - 1));
        if (i < 61 && i % 2 == 0 && v != t) return 1;  // powers of 4: exact
    }
    for (int j = 0; j < 256; ++j) {
        A[j] = (uint64_t)(exp2l(-(L)j / 256) * 0x1p62L + 0.5L);
        B[j] = j ? (uint64_t)(exp2l(-(L)j / 65536) * 0x1p63L + 0.5L) : (1ull << 63) - 1;
    }
    for (int i = 0; i < 300000; ++i) {
        double x = i % 2 ? (g() % 1000001) / 1e6 * 60 : exp2(-60 + (g() % 1000000) / 1e6 * 67);
        if (x == 0) x = 1;
        const double acc = x * x;
        const Dist d = dist_fix(dbits(acc));
        const L xt = sqrtl((L)acc), xv = ldexpl((L)d.X, d.q - 63);
        ed = fmaxl(ed, fabsl(xv / xt - 1));
        for (int n = 0; n < 3; ++n) {
            const Dist dd[1] = {d};
            int64_t v[1];
            matern_fix<1>(n, dd, A, B, v);
            ec[n] = fmaxl(ec[n], fabsl((L)v[0] * 0x1p-60L - corr(n, xt)));
        }
    }
    // Box-Muller pairs: rho^2 = -2 ln(1 - k1 2^-53), rho, cosine and sine of 2 pi k2 2^-53
    static SimTab T;
    const L hp = 1.570796326794896619231321691639751442L;
    for (int j = 0; j < 256; ++j) {
        const L x = (j + 0.5L) / 256;
        T.c[j] = (uint16_t)(j == 0 ? 32768 : j == 255 ? 16384 : (int)(32768 / (1 + x) + 0.5L));
        T.ln[j] = (int64_t)floorl(-logl((L)T.c[j] / 32768 * (j >= kLnHalf ? 2 : 1)) * 0x1p60L + 0.5L);
        T.cs[j] = (int64_t)(cosl(hp * x) * 0x1p62L + 0.5L);
        T.sn[j] = (int64_t)(sinl(hp * x) * 0x1p62L + 0.5L);
    }
    L ev = 0, eh = 0, et = 0;
    for (int i = 0; i < 300000; ++i) {
        uint64_t k1 = g() >> 11, k2 = g() >> 11;
        if (i % 5 == 0) k1 >>= g() % 53;                               // u1 near 1
        if (i % 7 == 0) k1 = (1ull << 53) - 1 - (k1 >> (g() % 53));    // u1 near 0
        if (i % 11 == 0) k2 = (g() % 9) << 50 & ((1ull << 53) - 1);    // eighths of a turn
        if (i == 1) k1 = 0;
        const Pair p = pair_fix(k1, k2, T);
        const L v = -2 * log1pl(-(L)k1 * 0x1p-53L), rho = sqrtl(v);
        ev = fmaxl(ev, fabsl((L)p.V * 0x1p-56L - v));
        eh = fmaxl(eh, fabsl(ldexpl((L)p.X, p.q - 63) - rho) * rho);
        const L a = 4 * hp * (L)k2 * 0x1p-53L;
        et = fmaxl(et, fmaxl(fabsl((L)p.cs * 0x1p-62L - cosl(a)), fabsl((L)p.sn * 0x1p-62L - sinl(a))));
    }
    printf("%Lg %Lg %Lg %Lg %Lg %Lg %Lg %Lg\n", er, ed, ev, eh, et, ec[0], ec[1], ec[2]);
    if (unit_fix(1.0) != 1ll << 60 || unit_fix(0.0) != 0) return 2;
    return 0;
}
"""


def test_fixed_point_functions(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    exe = tmp_path / "t"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
    er, ed, ev, eh, et, *ec = map(float, r.stdout.split())
    assert er <= 2.0 ** -58 and ed <= 2.0 ** -58, (er, ed)
    assert max(ec) <= 2.0 ** -55, ec
    # rho^2 in units 2^-56 from a logarithm within 2^-57, and no worse than an FP64 logarithm
    # (2^-54 of values near 1); the angle functions within a few units of 2^-62 times table products
    assert ev <= 2.0 ** -55 and eh <= 2.0 ** -55 and et <= 2.0 ** -58, (ev, eh, et)
