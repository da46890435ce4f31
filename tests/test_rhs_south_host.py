"""The integer-mantissa right-hand side where sin th < 0, compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_half_below_the_axis_is_the_mirror_image(tmp_path):
    """Taken (not handed to the FP64 form) and equal to the image's to the
    rounding of a result and of its terms: 4 x 2^-52."""
    exe = str(tmp_path / "rhs_south_host")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2602_07452_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "rhs_south_host.cu")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.returncode
    assert float(out.stdout) <= 4 * 2.0**-52, out.stdout
