"""Host check of fx_to_double (csrc/fixed_lap.cuh) over the whole range that the fixed-point windows
use, |L| < 2^63 (their sums reach 116 * 2^56): the correctly rounded binary64 value of
L * 2^(emax - 1080), for every position of the leading bit, ties and both ends of emax."""
import os
import random
import shutil
import subprocess
from fractions import Fraction as Fr

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2308_11469_gb300", "csrc")

PROBE = r"""
#include "fixed_lap.cuh"
#include <cstdio>
int main() {
    long long L;
    int e;
    while (std::scanf("%lld %d", &L, &e) == 2) std::printf("%a\n", helm::fx_to_double(L, e));
    return 0;
}
"""


def test_conversion_is_correctly_rounded_below_2_63(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)],
                   check=True)
    rng = random.Random(3)
    vals = [0, 1, -1, 2 ** 62, -2 ** 62, 2 ** 63 - 1, 1 - 2 ** 63, 116 * 2 ** 56, -116 * 2 ** 56, 27 * 2 ** 58]
    for b in range(63):
        for _ in range(40):
            v = (1 << b) | rng.getrandbits(b) if b else 1
            if b >= 53 and rng.random() < 0.5:         # a tie
                v = (v >> (b - 52) << (b - 52)) | (1 << (b - 53))
            vals.append(rng.choice((v, -v)))
    cases = [(v, e) for v in vals for e in (64, 65, 1023, 1080, 2029, 2030)]
    out = subprocess.run([str(exe)], input="".join(f"{v} {e}\n" for v, e in cases), capture_output=True, text=True,
                         check=True).stdout.split()
    assert len(out) == len(cases)
    for (v, e), got in zip(cases, out):
        assert float.fromhex(got) == float(Fr(v) * Fr(2) ** (e - 1080))
