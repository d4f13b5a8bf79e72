"""The preconditioner's panel (csrc/precond_layout.h, compiled for the host): every neighbourhood that
the product's kernel takes (14,464 points) has one that fits the shared memory of an SM."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORK = os.path.join(ROOT, "tests", "_build")   # git-ignored
CSRC = os.path.join(ROOT, "paper_2511_12450_gb300", "csrc")
MAIN = """#include <cstdio>
#include "precond_layout.h"
int main() {
    for (int q = 1; q <= 14464; ++q) std::printf("%d\\n", lfmm::pc_panel_columns(q));
}
"""


def test_panels_fit_shared_memory():
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a C++ compiler")
    os.makedirs(WORK, exist_ok=True)
    src, exe = os.path.join(WORK, "precond_panel.cpp"), os.path.join(WORK, "precond_panel")
    with open(src, "w") as f:
        f.write(MAIN)
    res = subprocess.run([cxx, "-std=c++17", "-I", CSRC, src, "-o", exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    cols = list(map(int, subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()))
    assert len(cols) == 14464 and cols[0] == 16
    for q, n in enumerate(cols, 1):
        # beside the kernel's own arrays: two 16 x 16 blocks of 16 bytes and some 120 bytes of reductions
        assert 0 <= n <= 16 and 16 * n * q + 2 * 16 * 16 * 16 + 128 <= 227 * 1024, q
