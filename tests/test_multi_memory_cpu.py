"""Device memory of grouped requests (tests/hostplan/memory_suite.cpp): without room for their
item map they run one by one, and serving's admission counts what they hold."""
import os
import subprocess

import numpy as np
import pytest

import test_hostplan_cpu as hostplan

CSRC = os.path.join(hostplan.ROOT, "paper_2108_04413_gb300", "csrc")


@pytest.fixture(scope="module")
def suite(tmp_path_factory):
    if not hostplan._have_toolchain():
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("memory") / "memory_suite")
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(hostplan.ROOT, "include"), "-I", CSRC, "-I",
                    hostplan.CUDA_INC, "-x", "c++", os.path.join(CSRC, "qf_api.cu"), "-x", "none",
                    os.path.join(hostplan.HERE, "pass_stub.cpp"), os.path.join(hostplan.HERE, "memory_suite.cpp"), "-o",
                    exe, "-lpthread"], check=True, timeout=600)
    return exe


def test_no_room_for_the_item_map(suite, tmp_path):
    hostplan._write_inputs(str(tmp_path))
    out = subprocess.run([suite, str(tmp_path)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    # no room: one by one, and again until the plan is made anew; then one grouped launch; nothing leaked
    assert out == ["0", "0", "0", "0", "0", "1", "0"]


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,rows", [(8, 64), (12, 8), (16, 2), (16, 32)])
def test_footprint_bounds_a_grouped_handle(suite, tmp_path, n, rows, dtype):
    """footprint_bytes bounds what a handle holds after a grouped call, and not by more than
    the 2.5 times it is held to without one."""
    from paper_2108_04413_gb300 import prep
    from paper_2108_04413_gb300.serving import footprint_bytes
    from workloads import amplitudes, integrals

    h, g = integrals(n // 2, 100 + n)
    T = prep.molecular_hamiltonian(h, g)
    A, exs = prep.uccsd_ansatz(n // 2, n // 2)
    T.tofile(tmp_path / "terms_fp.bin"), A.tofile(tmp_path / "ansatz_fp.bin")
    t = np.stack([amplitudes(len(exs), n + k, 0.1) for k in range(rows)]).astype(np.float64)
    t.tofile(tmp_path / "t_fp.bin")
    det = (1 << (n // 2)) - 1
    out = subprocess.run([suite, str(tmp_path), str(n), dtype, str(det), str(rows)], check=True, capture_output=True,
                         text=True, timeout=600).stdout.split()
    status, grouped, held = (int(v) for v in out)
    assert status == 0 and grouped == 1
    assert held <= footprint_bytes(n, dtype, det, A, len(T), rows) <= 2.5 * held


def test_server_charges_the_rows_it_groups():
    from paper_2108_04413_gb300 import prep
    from paper_2108_04413_gb300.serving import Server, System, footprint_bytes

    class Executor:
        run_multi = None

    A, _ = prep.uccsd_ansatz(4, 4)
    systems = {k: System(k, 8, 15, A, np.zeros(10)) for k in "ab"}
    for batch, qubits, rows in ((32, 16, 32), (32, 6, 1), (1, 16, 1)):
        srv = Server(systems, Executor(), workers=1, batch=batch, batch_qubits=qubits)
        assert srv._footprint("a") == footprint_bytes(8, "c64", 15, A, 10, rows)
        srv.close()
    assert footprint_bytes(8, "c64", 15, A, 10, 1) == footprint_bytes(8, "c64", 15, A, 10)
