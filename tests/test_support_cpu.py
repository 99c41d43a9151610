"""Circuits on a determinant as the C ABI plans them (passes over the reached tiles,
composite blocks alone and in passes, runs of one X mask), carried out on the host with
each launch's own index arithmetic, against the rotations one by one
(tests/hostplan/support_suite.cpp)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "hostplan")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
REPLACED = ("launch_zero_and_set", "launch_rot", "launch_tile", "launch_sparse")


@pytest.fixture(scope="module")
def suite(tmp_path_factory):
    if not (shutil.which("g++") and os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("support")
    csrc = os.path.join(ROOT, "paper_2108_04413_gb300", "csrc")
    cc = ["g++", "-O2", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I", CUDA_INC]
    subprocess.run(cc + [f"-D{k}=recorded_{k}" for k in REPLACED] + ["-c", os.path.join(HERE, "cuda_stub.cpp"), "-o",
                                                                    str(d / "stub.o")], check=True, timeout=600)
    subprocess.run(cc + ["-x", "c++", os.path.join(csrc, "qf_api.cu"), os.path.join(HERE, "support_suite.cpp"),
                         "-x", "none", str(d / "stub.o"), "-o", str(d / "suite"), "-lpthread"], check=True, timeout=600)
    return str(d / "suite")


def _run(suite, path, n, rots, dtype, written=()):
    from paper_2108_04413_gb300 import abi

    abi.as_rots(*(list(c) for c in zip(*rots))).tofile(path / "rots.bin")
    out = subprocess.run([suite, str(n), str((1 << n) // 3), dtype, str(path / "rots.bin"), *map(str, written)],
                         check=True, capture_output=True, text=True, timeout=600).stdout.split()
    return int(out[0]), float(out[1]), int(out[2]), int(out[3])


def _random(n, count, rng):
    out = []
    for k in range(count):
        q = rng.choice(n, size=int(rng.integers(1, 6)), replace=False)
        x = sum(1 << int(v) for v in q[: int(rng.integers(0, len(q) + 1))])
        out.append((x, int(rng.integers(0, 1 << n)), float(rng.uniform(-3.1, 3.1))))
    out[1] = ((1 << n) - 1, 5, 0.3)  # wider than a tile
    return out


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
@pytest.mark.parametrize("n,count", [(12, 40), (18, 4), (18, 24), (19, 12)])
def test_random_rotations(suite, tmp_path, n, count, dtype, tol):
    status, worst, parts, inner = _run(suite, tmp_path, n, _random(n, count, np.random.default_rng(n + count)), dtype)
    assert status == 0 and worst < tol
    assert (parts > 0) == (n >= 18)


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
@pytest.mark.parametrize("orbitals,masks", [(5, 400), (7, 70), (9, 60)])
def test_molecular_strings(suite, tmp_path, orbitals, masks, dtype, tol):
    from paper_2108_04413_gb300 import prep

    rng = np.random.default_rng(orbitals)
    h = rng.normal(size=(orbitals, orbitals))
    g = rng.normal(size=(orbitals,) * 4)
    g = g + g.transpose(1, 0, 2, 3)
    g = g + g.transpose(0, 1, 3, 2)
    g = g + g.transpose(2, 3, 0, 1)
    terms = prep.molecular_hamiltonian(h + h.T, g)
    terms = terms[np.isin(terms["x"], np.unique(terms["x"])[:masks])]
    rots = [(int(t["x"]), int(t["z"]), float(0.1 * t["coeff"])) for t in terms]
    status, worst, parts, inner = _run(suite, tmp_path, 2 * orbitals, rots, dtype)
    assert status == 0 and worst < tol
    assert (parts > 0) == (inner > 0) == (orbitals == 9)


@pytest.mark.parametrize("n", [12, 18])
@pytest.mark.parametrize("parity", [0, 1])
def test_runs_of_one_mask(suite, tmp_path, n, parity):
    rng = np.random.default_rng([n, parity])
    rots = []
    for x, count in ((0, 30), (3 << (n - 4), 24), (1, 300), (int(rng.integers(1, 1 << n)), 40), (0, 25)):
        while count:
            z = int(rng.integers(0, 1 << n))
            if x == 0 or bin(x & z).count("1") % 2 == parity:
                rots.append((x, z, float(rng.uniform(-3.1, 3.1))))
                count -= 1
    status, worst, *_ = _run(suite, tmp_path, n, rots, "c128")
    assert status == 0 and worst < 1e-12


def test_written_by_its_owner(suite, tmp_path):
    n = 18
    status, worst, parts, inner = _run(suite, tmp_path, n, _random(n, 10, np.random.default_rng(3)), "c128", ((1 << n) - 7,))
    assert status == 0 and worst < 1e-12
