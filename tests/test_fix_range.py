"""The limit of the data row's solved entries in the fixed-point factorisation, on the CPU: with it
no sum that the row takes part in leaves its range, whatever the data.  (A row of the factor has a
norm of at most 1; matrix entries hold +-8, the tensor cores' digit sums of order 0 and 1 are only
converted rightly below 2^22.)"""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_04477_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "bv_fix.cuh"
int main() { for (int n = 1; n <= 5000; ++n) printf("%d\n", bvfix::row_limit(n)); }
"""


def test_data_row_limit(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lims = [int(v) for v in subprocess.run([str(exe)], capture_output=True, text=True).stdout.split()]
    for n, g in enumerate(lims, 1):
        # the row's own entry, the columns before the panel and the panel's own, of which a value
        # below 1 may be used before it is found too large
        assert g >= 1 and (n ** 0.5) * 2.0 ** -g <= 4.0, (n, g)
        assert 2.0 ** -5 + ((n * 4.0 ** -g) + 16.0) ** 0.5 < 8.0, (n, g)
        assert g == 1 or (n ** 0.5) * 2.0 ** -(g - 1) > 4.0, (n, g)  # no tighter than that
    # digit sums of 16 columns: first digits of a data entry below 1/2, of a row of norm 1, and second
    # digits up to 512; order 1 of an unlimited data row (entries up to 1) would not fit
    norm = 512.0 + 2.0
    order1 = lambda top: 16 * top * 512.0 + 512.0 * 4.0 * norm
    assert order1(256.0) < 2 ** 22 < order1(512.0)
    assert 2 * 512.0 * 4.0 * norm < 2 ** 22
