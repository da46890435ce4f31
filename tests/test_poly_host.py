"""The bound of the deposit's per-cell polynomials, compiled for the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_a_bound_that_is_no_number_refuses_the_grid(tmp_path):
    """Cells so far out that the series is no number, before or after ones
    where the bound is met: the grid keeps the lattices."""
    exe = str(tmp_path / "poly_host")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2602_07452_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "poly_host.cu")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True)
    assert out.stdout.split() == ["1", "1", "0", "0"] * 2, out.stdout
