"""The solvers' fused vector passes: compiles tests/vectors_check.cu with the
library's kernels.cu and compares them bit for bit with the separate passes and
with the stated order of the dots, at the edges of blocks and grids."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1509_00216_gb300", "csrc")


def test_fused_vector_passes_keep_every_bit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "vectors_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
                    os.path.join(HERE, "vectors_check.cu"), os.path.join(CSRC, "kernels.cu"), "-o", exe], check=True)
    run = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout + run.stderr
