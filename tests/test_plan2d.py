"""The 2D step's choice between tiles and marched strips (csrc/plan.h, host
only) takes the faster one at FP32 shapes where both were measured and lie
more than 2 % apart."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1510_05061_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
needs_gxx = pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(os.path.join(CUDA, "include")),
                               reason="needs g++ and the CUDA headers")

PROGRAM = r"""
#include <cstdio>
#include "plan.h"
int main()
{
    int nx, ny, fp32, ppm;
    while (std::scanf("%d %d %d %d", &nx, &ny, &fp32, &ppm) == 4) {
        const hydro::Plan2D p = hydro::plan2d(nx, ny, fp32 != 0, ppm != 0);
        std::printf("%d %d %d\n", p.march, p.tx, p.ty);
    }
}
"""

# (nx, ny): threads of the fastest strip, or 0 where the tile is faster
FP32 = {(61, 61): 0, (384, 384): 0, (2600, 48): 0, (450, 450): 0, (600, 600): 0, (2600, 100): 0, (800, 700): 0,
        (40, 30000): 0, (64, 20000): 0, (256, 4000): 0, (160, 8000): 0, (250, 2600): 256, (360, 2600): 128,
        (1024, 1024): 128, (1448, 1448): 256, (2048, 2048): 128}


def plans(shapes, folder):
    """(threads of the strip or 0, tile) for each (nx, ny, fp32, ppm)."""
    src, exe = os.path.join(folder, "plan.cpp"), os.path.join(folder, "plan")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe], check=True)
    r = subprocess.run([exe], input="".join("%d %d %d %d\n" % s for s in shapes), capture_output=True, text=True, check=True)
    return [tuple(int(v) for v in line.split()) for line in r.stdout.splitlines()]


@needs_gxx
def test_the_faster_form_is_taken(tmp_path):
    for ((nx, ny), nt), got in zip(FP32.items(), plans([(nx, ny, 1, 0) for nx, ny in FP32], str(tmp_path))):
        assert (got[0] != 0) == (nt != 0), ((nx, ny), got)
        if (nx, ny) == (2048, 2048):
            assert got[0] == nt, got   # 101 us against 106 with the wider strip
