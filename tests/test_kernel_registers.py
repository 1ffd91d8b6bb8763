"""The FP32 tiles of the 2D step leave room for 48 resident warps per SM: large
grids are bound by instruction issue, and with 55 registers (32 warps) they
took a fifth longer.  The compiler's own report, no GPU needed."""

import os
import re
import shutil
import subprocess

import pytest

from paper_1510_05061_gb300 import build

UNIT = """
#include "step2d.cuh"
namespace hydro {
template __global__ void step2d_kernel<float, 32, 16, STAGE_HANCOCK, RECON_PLM>(const StepArgs);
template __global__ void step2d_kernel<float, 32, 16, STAGE_RK2, RECON_PLM>(const StepArgs);
template __global__ void step2d_kernel<float, 16, 16, STAGE_RK2, RECON_PPM>(const StepArgs);
}
"""


@pytest.mark.skipif(shutil.which(build._nvcc()) is None, reason="needs nvcc")
def test_fp32_2d_tiles_keep_their_warps(tmp_path):
    src = tmp_path / "unit.cu"
    src.write_text(UNIT)
    r = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-I", build.CSRC, "-Xptxas", "-v", "-c", str(src), "-o",
                        str(tmp_path / "unit.o")], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    used = [int(n) for n in re.findall(r"Used (\d+) registers", r.stderr)]
    assert len(used) == 3
    assert max(used) * 48 * 32 <= 65536, used   # registers of an SM
    assert not re.search(r"[1-9]\d* bytes spill", r.stderr)
