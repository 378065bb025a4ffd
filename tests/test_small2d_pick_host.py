"""Host check of the choice of a cluster size for the one-launch solves of small 2D grids
(csrc/launch.h): where a device cannot hold a form, the next smaller cluster takes its place, and
where it holds none the launch-by-launch path (0) does."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2308_11469_gb300", "csrc")

PROBE = r"""
#include "launch.h"
#include <cstdio>
int main() {
    for (int fits = 0; fits < 32; ++fits)
        for (int n : {15, 31, 63, 127})
            for (int c : {1, 12, 13, 32, 33, 96, 97})
                for (int m : {0, 1}) std::printf("%d %d %d %d %d\n", fits, n, c, m, helm::small2d_pick(n, c, m != 0, fits));
    return 0;
}
"""


def test_only_forms_that_fit_are_chosen(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)],
                   check=True)
    bit = {(63, 8): 1, (63, 4): 2, (63, 2): 4, (31, 4): 8, (31, 2): 16}
    rows = [tuple(map(int, r.split())) for r in
            subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 32 * 4 * 7 * 2
    for fits, n, count, mixed, cs in rows:
        wish = {63: 8 if count <= 12 else 4 if count <= 32 else 2, 31: 4 if count <= 32 else 2}.get(n, 0)
        sizes = [c for c in (8, 4, 2) if c <= wish and fits & bit.get((n, c), 0)]
        assert cs == (0 if count > (32 if mixed else 96) or not sizes else sizes[0])
