"""The integer form of the double to float conversion (csrc/lf_cvt.h), compiled
for the host, against the cast: every exponent with edge and random mantissas,
ties, the ends of the normal range, zeros, infinities and NaN."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1102_3094_gb300", "csrc")

PROGRAM = r"""
#include "lf_cvt.h"
#include <cstdio>
#include <cstring>
using namespace lf;
static uint64_t rng = 88172645463325252ull;
static uint64_t rnd() { rng ^= rng << 13; rng ^= rng >> 7; rng ^= rng << 17; return rng; }
static long bad = 0;
static void narrow_one(uint64_t u)
{
    double d; float f; uint32_t b, w;
    std::memcpy(&d, &u, 8);
    const int e = (int)(u >> 52 & 0x7ff);
    if (narrow_bits(u, &b) != (e >= 897 && e <= 1150)) { ++bad; return; }
    if (e < 897 || e > 1150) return;
    f = (float)d;
    std::memcpy(&w, &f, 4);
    if (b != w) ++bad;
}
int main()
{
    for (uint64_t s = 0; s < 2; ++s)
        for (uint64_t e = 0; e < 2048; ++e)
            for (int k = 0; k < 400; ++k) {
                uint64_t m = rnd() & 0xfffffffffffffull;
                if (k % 4 == 1) m = (m & ~0x1fffffffull) | 0x10000000;            // ties
                if (k % 4 == 2) m = (m & ~0x1fffffffull) | 0x0fffffff;
                if (k % 4 == 3) m = (m & ~0x1fffffffull) | 0x10000001;
                if (k == 0) m = 0;
                if (k == 4) m = 0xfffffffffffffull;
                if (k == 8) m = 0xffffff0000000ull;                               // carries into the exponent
                narrow_one(s << 63 | e << 52 | m);
            }
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_integer_conversion_equals_cast(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "cvt.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "cvt"
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
