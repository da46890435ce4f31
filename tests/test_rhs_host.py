"""The push's integer-mantissa right-hand side, compiled for the host: never
less accurate than the same formulas in double, over its ranges."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_integer_right_hand_side_against_long_double(tmp_path):
    """L2 relative error at most 1e-16 (one rounding, 2^-53 / sqrt 3 = 6.4e-17 at
    worst on average, and the 2^-57 of the chain; the FP64 form has 1.3e-16 to
    2.3e-16), the FP64 form's where that is smaller, and the refusals."""
    exe = str(tmp_path / "rhs_host")
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_2602_07452_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "rhs_host.cu")], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.returncode
    rows = [line.split() for line in out.stdout.splitlines()]
    assert len(rows) == 42
    for mode, i, x, d in rows:
        assert float(x) <= 1e-16 and float(x) <= 1.02 * float(d), (mode, i, x, d)
