"""Conversions between FP64 and block fixed point (hmg_fixed.cuh) on the host, subnormals included:
the scale of a value, the integer and back, against exact arithmetic."""
import os
import shutil
import subprocess

import pytest

from paper_1504_07499_gb300 import build

CODE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "hmg_fixed.cuh"
using namespace hmg::fx;
int main() {
    std::mt19937_64 g(1);
    long key = 0, fix = 0, cut = 0, back = 0;
    for (long i = 0; i < 400000; ++i) {
        // magnitudes 2^-890 .. 2^-1087: normal, subnormal, zero
        double d = std::ldexp((double)(long long)g(), -953 - (int)(g() % 198));
        if (i % 97 == 0) d = 0.0;
        int e;
        std::frexp(d, &e);
        const int E = key_of(d);
        key += E != (e < -1021 ? -1021 : d == 0.0 ? -1021 : e);   // zeros and subnormals share -1021
        // at the scale that a pencil of this value has it is held exactly
        const long long v = to_fixed(d, E - 58);
        fix += d == 0.0 ? v != 0 : std::ldexp((double)v, E - 58) != d;
        if (d != 0.0) {   // at a coarser one to half a unit
            const int c = E - 58 + (int)(g() % 70);
            cut += std::fabs((double)to_fixed(d, c) - std::ldexp(std::ldexp(d, 600), -c - 600)) > 0.5 + 1e-9;
        }
        // back: nearest double, 2^-1074 apart below 2^-1022
        const long long w = (long long)g() >> (g() % 64);
        const int x = -1200 + (int)(g() % 260);
        const double f = is_low(x) ? from_fixed<true>(w, x) : from_fixed(w, x);
        const double n = std::ldexp((double)w, x);   // rounds once or twice: at most one unit from f
        back += std::fabs(f - n) > std::fmax(std::ldexp(1.0, -1074), std::ldexp(std::fabs(n), -52));
    }
    std::printf("%ld %ld %ld %ld\n", key, fix, cut, back);
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"), reason="no nvcc")
def test_conversions(tmp_path):
    (tmp_path / "t.cu").write_text(CODE)
    exe = str(tmp_path / "t")
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, str(tmp_path / "t.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0", "0", "0"]
