"""Expectation values of general states through passes over shared-memory tiles.

On the CPU the plan's passes are evaluated with the kernel's index arithmetic
(tests/hostplan/pass_suite.cpp) against the oracle; on the GPU the kernels are
compared with the allocation-free call, which takes the per-group kernel, and
with the oracle's definition.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests", "hostplan")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def _terms(n, count, rng, heavy=True):
    """Random strings, with the diagonal group, groups of many terms, odd-Y and
    repeated terms, masks on the lowest and highest qubits and (heavy) X masks too
    wide for a tile."""
    from paper_2108_04413_gb300.abi import as_terms

    x = rng.integers(0, 1 << n, count) & rng.integers(0, 1 << n, count) & rng.integers(0, 1 << n, count)
    z = rng.integers(0, 1 << n, count)
    x[:6], x[6:20], x[20:26] = 0, x[30], x[31] | 1
    x[26], x[27], x[28], z[29], x[29] = 1, 1 << (n - 1), 1 | 1 << (n - 1), 0, 3
    z[20], x[33], z[33] = z[21], x[32], z[32]
    if heavy:
        x[34:37] = (1 << n) - 1 - np.array([0, 1, 2])
    return as_terms(x.astype(np.uint64), z.astype(np.uint64), rng.normal(size=count) / np.sqrt(count))


def _expect(psi, T):
    b = np.arange(len(psi), dtype=np.uint64)
    total = 0.0
    for x, z, c in zip(T["x"], T["z"], T["coeff"]):
        v = np.vdot(psi, 1j ** int(np.bitwise_count(x & z)) * (1.0 - 2.0 * (np.bitwise_count(z & (b ^ x)) & 1))
                    * psi[(b ^ x).astype(np.int64)])
        total += c * v.real
    return total


@pytest.fixture(scope="module")
def suite(tmp_path_factory):
    if not (shutil.which("g++") and os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("passes") / "pass_suite")
    csrc = os.path.join(ROOT, "paper_2108_04413_gb300", "csrc")
    cmd = ["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I", CUDA_INC,
           "-x", "c++", os.path.join(csrc, "qf_api.cu"), "-x", "none", os.path.join(HERE, "pass_suite.cpp"),
           "-o", exe, "-lpthread"]
    subprocess.run(cmd, check=True, capture_output=True, timeout=600)
    return exe


@pytest.mark.parametrize("n,dtype,count", [(15, "c128", 140), (15, "c128", 400), (15, "c64", 140), (16, "c64", 300)])
def test_passes_cover_every_pair_once(suite, tmp_path, n, dtype, count):
    from workloads import random_state

    T = _terms(n, count, np.random.default_rng(n + count))
    psi = random_state(n, 5).astype(np.complex128 if dtype == "c128" else np.complex64)
    T.tofile(tmp_path / "terms.bin"), psi.tofile(tmp_path / "state.bin")
    out = subprocess.run([suite, str(tmp_path), str(n), dtype], capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stdout
    value, passes, rest = out.stdout.split()
    ref = _expect(psi.astype(np.complex128), T)
    assert int(passes) >= 1 and int(rest) == len({int(x) for x in T["x"] if int(x) >> (3 if dtype == "c128" else 4)
                                                  and bin(int(x) >> (3 if dtype == "c128" else 4)).count("1") > 9})
    assert abs(float(value) - ref) < 1e-12  # FP64 sums of ~n terms of a unit vector


@pytest.mark.gpu
@pytest.mark.parametrize("n,count", [(15, 140), (15, 700), (17, 40), (20, 400)])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-13), ("c64", 2e-6)])
def test_passes_match_the_group_kernel(n, count, dtype, tol):
    import torch

    from paper_2108_04413_gb300 import qf
    from workloads import random_state

    T = _terms(n, count, np.random.default_rng(n + count))
    psi = random_state(n, 7).astype(np.complex128 if dtype == "c128" else np.complex64)
    st = qf.State(n, dtype)
    st.from_numpy(psi)
    v = st.expectation(T)[0]
    assert v == st.expectation(T)[0]  # fixed summation order
    dev = torch.from_numpy(psi).cuda()
    ref = qf.expectation_noalloc(dev.data_ptr(), n, dtype, torch.cuda.current_stream().cuda_stream, T)[0]
    # sum |coeff| <= sqrt(count): FP64 (FP32) rounding of a unit vector's pair products
    assert abs(v - ref) < tol
    if n <= 15:
        assert abs(v - _expect(psi.astype(np.complex128), T)) < tol
