"""The reciprocal and the reciprocal root that the float64 leaves and rotations use
in place of a division and CUDA's rsqrt (csrc/df_arith.cuh), over the whole range
of exponents, by tests/df_arith_check.cu."""
import os
import subprocess

import pytest

from paper_1607_06303_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_reciprocals(gpu_lib, tmp_path):
    exe = str(tmp_path / "df_arith_check")
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I", build.CSRC,
                   os.path.join(ROOT, "tests", "df_arith_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert out.stdout.startswith("ok ")
