"""A grouped request of very many blocks: the item counts of 17,550 blocks do not fit beside a
sector that takes most of a CTA's shared memory (20 qubits, 5 alpha and 2 beta electrons,
complex128: 181 KB of psi and lambda)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()

from paper_2108_04413_gb300 import prep, qf  # noqa: E402
from workloads import amplitudes, integrals  # noqa: E402


def test_many_blocks_in_a_large_sector():
    h, g = integrals(10, 3)
    one, exs = prep.uccsd_ansatz(10, 7)
    copies = 25  # the operators repeated, each repetition with its own parameters
    A = np.concatenate([one] * copies)
    A["param"] += np.repeat(np.arange(copies) * len(exs), len(one)).astype(A["param"].dtype)
    n_par = copies * len(exs)
    assert n_par > 17000
    det = sum(1 << 2 * k for k in range(5)) | sum(2 << 2 * k for k in range(2))
    T = prep.molecular_hamiltonian(h, g)
    t = np.stack([amplitudes(n_par, 7 + k, 0.02) for k in range(2)])
    st = qf.State(20, "c128")
    e1, g1 = st.energy_grad(det, A, t[1], T)
    qf.kernel_launches(True)
    e, gr = st.energy_grad_multi(det, A, t, T)
    assert qf.kernel_launches(True) == 2  # the grouped evaluation and the reset to |det>
    # 17,550 blocks of two roundings each on a unit vector
    assert abs(e[1] - e1) < 1e-11 and np.abs(gr[1] - g1).max() < 1e-10
    st.close()
