"""The mixed form's p.q and r.z are finished from FP32 pairs without the FP64
pipe (Sum3 in csrc/spfd_reduce.cuh).  Host check (tests/pair_sum_check.cu):
each sum within its derived bound, and no further from the exact sum, in the
mean over the cases, than FP64 additions of the same pairs."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2010_12879_gb300", "csrc")


def test_pair_sums_are_as_accurate_as_fp64_additions(tmp_path):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "pair_sum_check")
    b = subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include"),
                        "-I" + CSRC, os.path.join(HERE, "pair_sum_check.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert b.returncode == 0, b.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
    word, cases, e3, e64 = r.stdout.split()
    assert word == "ok" and int(cases) == 128
    assert float(e3) <= float(e64)


def test_finishing_kernel_adds_in_three_parts():
    text = open(os.path.join(CSRC, "spfd_krylov.cu")).read()
    body = text[text.index("k_finish_pairs(const double"):]
    body = body[:body.index("\n}\n")]
    assert "sum3_add(a[k], q.x, q.y, 0.f);" in body and "two_sum_add(" not in body
