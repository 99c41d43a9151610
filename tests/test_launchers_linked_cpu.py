"""The compiled planner needs every kernel launcher: no reference to one is weak, so a library
linked without a kernel file does not load."""
import os
import shutil
import subprocess

import pytest

from paper_2108_04413_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_launchers_are_ordinary_symbols(tmp_path):
    nvcc = build._nvcc()
    if not (shutil.which("nm") and (os.path.exists(nvcc) or shutil.which(nvcc))):
        pytest.skip("needs nvcc and nm")
    obj = str(tmp_path / "qf_api.o")
    subprocess.run([nvcc, *build.ARCH, "-O0", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-c",
                    os.path.join(build.CSRC, "qf_api.cu"), "-o", obj], check=True, timeout=600)
    names = subprocess.run(["nm", "-C", "--undefined-only", obj], check=True, capture_output=True, text=True).stdout
    launchers = [line.split()[0] for line in names.splitlines() if "qf::launch_" in line]
    assert len(launchers) > 20 and set(launchers) == {"U"}


def test_every_path_plans_with_every_launcher(tmp_path):
    """The planner's suite on the complete test double: every path plans, twice the same, and
    no device memory is left."""
    import test_hostplan_cpu as hostplan

    if not hostplan._have_toolchain():
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "plan_suite")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                    "-I", hostplan.CUDA_INC, "-x", "c++", os.path.join(build.CSRC, "qf_api.cu"), "-x", "none",
                    *(os.path.join(hostplan.HERE, f) for f in ("cuda_stub.cpp", "pass_stub.cpp", "plan_suite.cpp")),
                    "-o", exe, "-lpthread"], check=True, timeout=600)
    hostplan._write_inputs(str(tmp_path))
    rows = hostplan._run((exe, str(tmp_path)))
    assert len(rows) == 17 and all(status == 0 and copies > 0 for status, copies, _, _ in rows.values())
    assert rows == hostplan._run((exe, str(tmp_path)))
