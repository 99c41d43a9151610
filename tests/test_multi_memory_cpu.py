"""Grouped requests where the device has no room for their item map run one by one
(tests/hostplan/memory_suite.cpp)."""
import os
import subprocess

import pytest

import test_hostplan_cpu as hostplan

CSRC = os.path.join(hostplan.ROOT, "paper_2108_04413_gb300", "csrc")


def test_no_room_for_the_item_map(tmp_path):
    if not hostplan._have_toolchain():
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "memory_suite")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(hostplan.ROOT, "include"), "-I", CSRC, "-I",
                    hostplan.CUDA_INC, "-x", "c++", os.path.join(CSRC, "qf_api.cu"), "-x", "none",
                    os.path.join(hostplan.HERE, "pass_stub.cpp"), os.path.join(hostplan.HERE, "memory_suite.cpp"), "-o",
                    exe, "-lpthread"], check=True, timeout=600)
    hostplan._write_inputs(str(tmp_path))
    out = subprocess.run([exe, str(tmp_path)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    # no room: one by one, and again until the plan is made anew; then one grouped launch; nothing leaked
    assert out == ["0", "0", "0", "0", "0", "1", "0"]
