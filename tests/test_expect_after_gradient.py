"""A Hamiltonian planned by a gradient call, which keeps no masks for expectation passes, gives
the passes of a fresh plan (tests/hostplan/late_suite.cpp on the CPU; the kernels on the GPU)."""
import os
import subprocess

import numpy as np
import pytest

import test_expect_passes as passes
from test_hostplan_cpu import _have_toolchain


@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_passes_after_a_gradient(tmp_path, dtype):
    from workloads import random_state

    if not _have_toolchain():
        pytest.skip("needs g++ and the CUDA headers")
    exe, csrc = str(tmp_path / "late_suite"), os.path.join(passes.ROOT, "paper_2108_04413_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(passes.ROOT, "include"), "-I", csrc, "-I",
                    passes.CUDA_INC, "-x", "c++", os.path.join(csrc, "qf_api.cu"), "-x", "none",
                    os.path.join(passes.HERE, "late_suite.cpp"), "-o", exe, "-lpthread"], check=True, timeout=600)
    n = 15
    T = passes._terms(n, 140, np.random.default_rng(9))
    psi = random_state(n, 5).astype(np.complex128 if dtype == "c128" else np.complex64)
    T.tofile(tmp_path / "terms.bin"), psi.tofile(tmp_path / "state.bin")
    out = subprocess.run([exe, str(tmp_path), str(n), dtype], check=True, capture_output=True, text=True, timeout=600)
    fresh, late, npass, rest = out.stdout.split()
    assert fresh == late and int(npass) >= 1 and int(rest) >= 1


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_passes_after_a_gradient_gpu(dtype):
    from paper_2108_04413_gb300 import abi, qf
    from workloads import random_state

    n = 17
    T = passes._terms(n, 200, np.random.default_rng(3))
    psi = random_state(n, 7).astype(np.complex128 if dtype == "c128" else np.complex64)
    a, b = qf.State(n, dtype), qf.State(n, dtype)
    b.energy_grad(1, abi.as_arots(np.array([3], np.uint64), np.array([4], np.uint64), np.array([0.5]),
                                  np.array([0])), np.array([0.3]), T)
    a.from_numpy(psi), b.from_numpy(psi)
    assert a.expectation(T)[0] == b.expectation(T)[0]  # fixed summation order
    a.close(), b.close()
