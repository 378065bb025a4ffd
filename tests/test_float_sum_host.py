"""Host check of the float sums of the complex64 residual norms (csrc/float_sum.cuh), compiled for
the CPU and compared with exact rationals: eight warps' sums, of any spread, up to and beyond the
floats' range, are added as accurately as in FP64.  One rounding of 2^-53 and, in the two lower
floats, less than 2^-66 of the sum."""
import math
import os
import shutil
import subprocess
from fractions import Fraction as Fr

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2308_11469_gb300", "csrc")

PROBE = r"""
#include "float_sum.cuh"
#include <cmath>
#include <cstdio>
#include <random>
int main() {
    std::mt19937_64 g(7);
    std::uniform_real_distribution<float> U(0.5f, 0.999f);
    for (int t = 0; t < 20000; ++t) {
        float v[8];
        const int top = t % 4 == 0 ? 127 : (int)(g() % 247) - 120, spread = 1 + (int)(g() % (t % 3 ? 60 : 3));
        for (int i = 0; i < 8; ++i) {
            v[i] = std::ldexp(U(g), 1 + top - (int)(g() % spread));
            if (g() % 30 == 0) v[i] = 0.f;
        }
        for (int i = 0; i < 8; ++i) std::printf("%a ", (double)v[i]);
        std::printf("%a\n", helm::sum_floats(v, 8));
    }
    const float bad[3] = {INFINITY, NAN, 1.f};
    std::printf("%a %a\n", helm::sum_floats(bad, 1), helm::sum_floats(bad + 1, 2));
    return 0;
}
"""


def test_sums_are_rounded_once(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()
    last = [float.fromhex(x) for x in out.pop().split()]
    assert math.isinf(last[0]) and math.isnan(last[1])
    assert len(out) == 20000
    beyond = 0
    for line in out:
        v = [Fr(float.fromhex(x)) for x in line.split()]
        want, got = sum(v[:8]), v[8]
        if want >= 2 ** 128:                  # (in FP64, one by one)
            beyond += 1
            assert abs(got - want) <= 7 * want / 2 ** 53
        else:
            assert abs(got - want) <= want * (Fr(1, 2 ** 53) + Fr(1, 2 ** 66))
    assert beyond > 1000
