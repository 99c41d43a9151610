"""Runs of one X mask (one rotation by the signed sum of their angles) at angles far past pi,
against the rotations one by one: on the CPU as planned, with the device's sums
(tests/hostplan/circuit_suite.cpp), and on the GPU.

Tolerance: a rotation rounds an amplitude by about 1e-16, so a few hundred rotations one by
one are off by about 1e-14 at most; a run's own phase is off by less.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "hostplan")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
REPLACED = ("launch_zero_and_set", "launch_rot", "launch_tile", "launch_sparse")
TOL = 1e-13


@pytest.fixture(scope="module")
def suite(tmp_path_factory):
    if not (shutil.which("g++") and os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("circuit")
    csrc = os.path.join(ROOT, "paper_2108_04413_gb300", "csrc")
    cc = ["g++", "-O2", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I", CUDA_INC]
    subprocess.run(cc + [f"-D{k}=recorded_{k}" for k in REPLACED] + ["-c", os.path.join(HERE, "cuda_stub.cpp"), "-o",
                                                                    str(d / "stub.o")], check=True, timeout=600)
    subprocess.run(cc + ["-x", "c++", os.path.join(csrc, "qf_api.cu"), os.path.join(HERE, "circuit_suite.cpp"),
                         "-x", "none", str(d / "stub.o"), "-o", str(d / "suite"), "-lpthread"], check=True, timeout=600)
    return str(d / "suite")


def _run(suite, path, n, rots, dtype, written=()):
    rots.tofile(path / "rots.bin")
    out = subprocess.run([suite, str(n), str((1 << n) // 3), dtype, str(path / "rots.bin"), *map(str, written)],
                         check=True, capture_output=True, text=True, timeout=600).stdout.split()
    return int(out[0]), float(out[1]), int(out[2]), int(out[3])


def _runs(n, largest, parity, rng):
    """Diagonal runs and runs of one X mask (strings of one parity of Y letters commute)."""
    from paper_2108_04413_gb300 import abi

    rots = []
    for x, count in ((0, 38), (1, 256), (3 << (n - 4), 24), (int(rng.integers(1, 1 << n)), 38), (0, 257)):
        while count:
            z = int(rng.integers(0, 1 << n))
            if x == 0 or bin(x & z).count("1") % 2 == parity:
                rots.append((x, z, largest * float(rng.uniform(-1, 1))))
                count -= 1
    rots.insert(38, ((1 << n) - 1, 5, 0.3))  # the first run acts on more than one determinant afterwards
    return abi.as_rots(*(list(c) for c in zip(*rots)))


@pytest.mark.parametrize("n,parity,largest", [(11, p, a) for p in (0, 1) for a in (3.14, 100.0, 1e6, 1e12, 1e15, 1e308)]
                         + [(18, 1, 1e6)])
def test_large_angles_as_planned(suite, tmp_path, n, parity, largest):
    rots = _runs(n, largest, parity, np.random.default_rng([n, parity]))
    status, worst, *_ = _run(suite, tmp_path, n, rots, "c128")
    assert status == 0 and worst < TOL


@pytest.mark.gpu
@pytest.mark.parametrize("n,parity", [(11, 0), (19, 1)])
@pytest.mark.parametrize("largest", [3.14, 1e6, 1e12, 1e308])
def test_large_angles_one_by_one(n, parity, largest):
    from paper_2108_04413_gb300 import qf

    rots = _runs(n, largest, parity, np.random.default_rng([n, parity, 1]))
    st, ref = qf.State(n, "c128"), qf.State(n, "c128")
    st.set_basis((1 << n) // 3), ref.set_basis((1 << n) // 3)
    st.apply_circuit(rots)
    for r in rots:
        ref.apply_pauli_exp(int(r["x"]), int(r["z"]), float(r["theta"]))
    d = np.abs(st.to_numpy() - ref.to_numpy())
    assert np.isfinite(d).all() and d.max() < TOL
