"""Expectation values where the device has no room for the passes' tables: the per-group kernel,
planned once and not on every call (tests/hostplan/full_suite.cpp)."""
import os
import subprocess

import numpy as np
import pytest

import test_expect_passes as passes
from test_hostplan_cpu import _have_toolchain


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_no_room_for_pass_tables(tmp_path, dtype):
    from workloads import random_state

    if not _have_toolchain():
        pytest.skip("needs g++ and the CUDA headers")
    exe, csrc = str(tmp_path / "full_suite"), os.path.join(passes.ROOT, "paper_2108_04413_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(passes.ROOT, "include"), "-I", csrc, "-I",
                    passes.CUDA_INC, "-x", "c++", os.path.join(csrc, "qf_api.cu"), "-x", "none",
                    os.path.join(passes.HERE, "full_suite.cpp"), "-o", exe, "-lpthread"], check=True, timeout=600)
    n = 15
    passes._terms(n, 140, np.random.default_rng(9)).tofile(tmp_path / "terms.bin")
    random_state(n, 5).astype(np.complex128 if dtype == "c128" else np.complex64).tofile(tmp_path / "state.bin")
    out = subprocess.run([exe, str(tmp_path), str(n), dtype], check=True, capture_output=True, text=True, timeout=600)
    taken, made = ([int(v) for v in out.stdout.split()[k:8:2]] for k in (0, 1))
    assert taken[:3] == [0, 0, 0] and taken[3] >= 1 and out.stdout.split()[8] == "1"
    # the first call plans the passes; the next ones only ask for room
    assert made[0] > 10 and made[1] == made[2] == 0 and made[3] > 10
