"""The kernels' harmonic constants, which the compiler builds, against 40 digits rounded once."""
import subprocess

import mpmath
import numpy as np

from paper_2609_05709_b200 import build

PROGRAM = r"""
#include <cstdio>
#include "harmonic_tables.h"
int main() {
    constexpr soap::HarmonicTables t = soap::harmonic_tables();
    for (int i = 0; i < soap::kHarmonicTerms; ++i) printf("%a %a %a %a %a %a\n", t.norm[i], t.norm_lm[i], t.step[i][0], t.step[i][1], t.step[i][2], t.step[i][3]);
    for (int m = 0; m <= soap::kHarmonicL; ++m) printf("%a\n", t.dfact[m]);
}
"""


def test_every_entry_is_the_rounded_value(tmp_path):
    (tmp_path / "tables.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.CSRC, str(tmp_path / "tables.cpp"), "-o", str(tmp_path / "tables")], check=True)
    lines = subprocess.run([str(tmp_path / "tables")], check=True, capture_output=True, text=True).stdout.splitlines()
    got = [[np.float32(float.fromhex(v)) for v in line.split()] for line in lines]
    f = np.float32
    with mpmath.workdps(40):
        at = 0
        for l in range(13):
            for m in range(l + 1):
                a = mpmath.sqrt(mpmath.mpf(2 * l + 1) / (4 * mpmath.pi) * mpmath.factorial(l - m) / mpmath.factorial(l + m) * (2 if m else 1))
                a = f(float(a))
                want = [a, f(l + m) * a, f(2 * l + 1) / f(l + 1 - m), f(l + m) / f(l + 1 - m)]
                want += [f(2 * l + 1) / f(l - m), f(l + m + 1) / f(l - m)] if l > m else [f(0), f(0)]
                assert got[at] == want, (l, m)
                at += 1
        for m in range(13):
            assert got[at + m] == [f(float(mpmath.fac2(2 * m - 1)))], m
