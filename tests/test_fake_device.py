"""Host-side handling of device resources, against a fake CUDA runtime (no GPU):
compiles tests/fake_device_check.cpp, whose runtime functions take the place of
the real ones in the library, and runs its cases."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
PACKAGE = os.path.join(ROOT, "paper_1509_00216_gb300")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def check(mpslcc, tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fake") / "fake_device_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-rdynamic", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(PACKAGE, "csrc"), "-isystem", os.path.join(CUDA, "include"),
                    os.path.join(HERE, "fake_device_check.cpp"), os.path.join(PACKAGE, "libmpslcc.so"),
                    "-Wl,-rpath," + PACKAGE, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("case", ["idle_memory", "failed_create", "refused_buffer"])
def test_device_resources(check, case):
    run = subprocess.run([check, case], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, run.stdout + run.stderr
