"""FP64 products (gemm_f64.cu) term by term: compiles tests/f64_products_check.cu
with the library's kernels and holds every output to the error bound of a chain
of FP64 fused multiply-adds over its terms -- operands graded in opposite
directions, unit rows over noise, rows near the end of the range, several
scaling blocks, K runs -- on every kernel that the plan can choose."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1509_00216_gb300", "csrc")


def _check(tmp_path, mode):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "f64_products_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", CSRC, os.path.join(HERE, "f64_products_check.cu"),
                    os.path.join(CSRC, "gemm_f64.cu"), "-o", exe], check=True)
    run = subprocess.run([exe, mode], capture_output=True, text=True, timeout=600)
    assert run.returncode == 0, run.stdout + run.stderr


def test_the_cases_reach_every_kernel(tmp_path):
    _check(tmp_path, "plan")


@pytest.mark.gpu
def test_every_output_is_within_the_bound_of_a_multiply_add_chain(tmp_path):
    _check(tmp_path, "run")
