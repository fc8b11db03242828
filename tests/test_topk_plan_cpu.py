"""The plan arithmetic of the exact top-k (csrc/topk_plan.cuh), compiled for the host from
the library's own sources (tests/native/topk_plan_check.cu)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_13601_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is not available")
    out = str(tmp_path_factory.mktemp("plan") / "topk_plan_check")
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-gencode",
                           "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           os.path.join(ROOT, "tests", "native", "topk_plan_check.cu"),
                           "-o", out])
    return out


@pytest.mark.parametrize("check", ["claims", "rows", "admitted", "table"])
def test_plan_arithmetic(exe, check):
    out = subprocess.run([exe, check], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout == "ok\n"
