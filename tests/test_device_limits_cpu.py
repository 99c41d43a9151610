"""A kernel's shared-memory limit is raised on every device that launches it, once on each
(tests/hostplan/device_suite.cpp), and by every launcher that way."""
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_04413_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def test_limit_is_raised_on_each_device(tmp_path):
    if not (shutil.which("g++") and os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "device_suite")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "hostplan", "device_suite.cpp"), "-o", exe, "-lpthread"], check=True,
                   timeout=600)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    # devices 0 and 1 once, 2 again after its failure, 63 once, 70 (past the flags) on every call
    assert out == ["3", "0", "1,1", "1,1", "2,2", "1,1", "2,2", "0", "0"]


def test_launchers_raise_it_per_device():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        assert "cudaFuncSetAttribute" not in open(path).read(), path
