"""The rule for a tree's depth (csrc/fmm_internal.h), compiled for the host: down to the
levels of the device builder's grids a level wants 44 nodes a box, beyond them, where the
host builds the tree, 64; level 3 and handles for differentiation 64 throughout."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include <cstdio>
#include "fmm_internal.h"
int main() {
    gnk::Boundary b;
    for (int diff = 0; diff < 2; ++diff) {
        b.diff = diff;
        for (int l = 3; l <= 13; ++l)
            for (int mean = 20; mean <= 70; mean += 1)
                std::printf("%d %d %d %d\n", diff, l, mean, (int)gnk::fmm_level_wanted(b, l, mean, 2.0 * mean));
    }
    std::printf("%d\n", gnk::kMaxGridLevel);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")),
                    reason="needs g++ and the CUDA headers")
def test_levels_wanted(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"),
                    "-I", os.path.join(ROOT, "paper_1308_5351_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    deepest = int(lines[-2])
    assert deepest == 11
    for line in lines[:-2]:
        diff, l, mean, wanted = map(int, line.split())
        old = mean >= 64
        if diff or l == 3 or l > deepest:
            assert wanted == old, line
        else:  # 44, or the geometric mean with the level above (here twice the nodes) 62
            assert wanted == (mean >= 44 or (mean >= 28 and 2 * mean * mean >= 62 * 62)), line
