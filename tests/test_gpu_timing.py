"""Every kernel that a call launches is in one of the kernel timings: circuits on a determinant
(which also check the state they read in part), a Trotter step, an expectation value, an ansatz
without sector form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()

from paper_2108_04413_gb300 import abi, prep, qf  # noqa: E402
from workloads import integrals  # noqa: E402


def _circuit(n):
    R = prep.random_circuit(n, 40, 1)
    return lambda st: (st.set_basis(3), st.apply_circuit(R))


def _trotter(n):
    h, g = integrals(n // 2, 1)
    T = prep.molecular_hamiltonian(h, g)
    return lambda st: (st.set_basis(3), st.trotter(T, 0.1, 1))


def _expectation(n):
    T = prep.random_hamiltonian(n, 100, 1)
    return lambda st: (st.apply_pauli_exp(1, 0, 0.3), st.expectation(T))


def _gradient(n):
    R = prep.random_circuit(n, 30, 2)
    A = abi.as_arots(R["x"], R["z"], np.ones(len(R)), np.arange(len(R)))
    T = prep.random_hamiltonian(n, 50, 2)
    return lambda st: st.energy_grad(3, A, R["theta"], T)


@pytest.mark.parametrize("work", [_circuit, _trotter, _expectation, _gradient])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_timed_launches_are_all_launches(work, dtype):
    n = 18
    run, st = work(n), qf.State(n, dtype)
    run(st)  # plans
    torch.cuda.synchronize()
    qf.kernel_launches(True)
    qf.profile_begin(qf.K_ALL)
    run(st)
    torch.cuda.synchronize()
    timed, ms = qf.profile_read(qf.K_ALL)
    qf.profile_end()
    assert timed == qf.kernel_launches(True) > 0 and ms > 0
    st.close()
