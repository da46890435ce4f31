"""The integer-mantissa reciprocal and reciprocal square root, compiled for the
host, with FP32 estimates as far off as the hardware's may be."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_reciprocals_with_estimates_moved_by_two_ulp(tmp_path):
    """At the ends of the mantissa's range (where a moved estimate leaves
    [1/2, 1)) and over random draws: the series' omitted terms (e^3 of e below
    2^-21: 2^-63) and the units of its 60 fraction bits dropped by four integer
    products, each at most a few of 2^-60: 16 of them."""
    exe = str(tmp_path / "xf_host")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2602_07452_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "xf_host.cu")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True)
    worst = [float(x) for x in out.stdout.split()]
    assert len(worst) == 2 and max(worst) <= 16.0, worst
