"""The rule that chooses the fused step's tiles (host code, run on the CPU): what it
chooses is what is launched, and can be."""
import os
import subprocess

import pytest

from paper_2605_12915_gb300 import _build

SIZES = [(2, 2), (8, 4), (40, 38), (96, 96), (256, 256), (333, 250), (352, 352), (383, 400),
         (384, 384), (320, 432), (416, 320), (448, 320), (512, 512), (640, 608), (1024, 1024),
         (1021, 1024), (2048, 2048), (2, 1048592), (16, 1048592), (16, 2097120), (40, 700000)]
SOURCE = r"""
#include "af_launch.cuh"
#include <cstdio>
using namespace af;
int main() {
  int nx, ny;
  while (std::scanf("%d %d", &nx, &ny) == 2) {
    StepArgs<float> a = {};
    a.nx = nx;
    a.ny = ny;
    const int g = choose_step_geometry(a, 152);
    std::printf("%d %d %d %d %d\n", STEP_GEOMS[g].tx, STEP_GEOMS[g].ty, STEP_GEOMS[g].pipe,
                (int)pipe_eligible(a), (int)pipe_eligible(a, STEP_GEOMS[g].ty));
  }
}
"""


@pytest.mark.slow
def test_the_choice_can_be_and_is_launched(tmp_path):
    src, exe = tmp_path / "choice.cu", tmp_path / "choice"
    src.write_text(SOURCE)
    subprocess.check_call([_build.nvcc(), "-std=c++17", *_build.ARCH, "-I", _build.CSRC, str(src),
                           "-o", str(exe)])
    out = subprocess.run([str(exe)], input="\n".join("%d %d" % s for s in SIZES), text=True,
                         stdout=subprocess.PIPE, check=True).stdout.split("\n")
    for (nx, ny), line in zip(SIZES, out):
        tx, ty, pipe, takes_32x32, takes = map(int, line.split())
        if pipe:
            assert takes, (nx, ny)
        else:  # rows of tiles are a launch's y dimension
            assert -(-ny // ty) <= 65535, (nx, ny)
        # a grid on 32 x 32 tiles runs the persistent kernel wherever that takes it
        if (tx, ty) == (32, 32):
            assert pipe == takes_32x32, (nx, ny)
