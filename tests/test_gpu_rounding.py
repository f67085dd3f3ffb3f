"""sqrt_rn and recip_rn round correctly: every bit equal to CUDA's sqrt() and
division on 2^25 values (tests/rounding_check.cu)."""

import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_sqrt_and_reciprocal_round_correctly(tmp_path):
    from paper_2010_12879_gb300 import build
    exe = str(tmp_path / "rounding_check")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS,
                    os.path.join(HERE, "rounding_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["recip", "0", "sqrt", "0"]
