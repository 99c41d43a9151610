"""Grouped small requests at the edges of their launch shapes: more requests than SMs
(two per SM), and a sector whose state takes most of a CTA's shared memory and whose
blocks have more items than two rounds of the step threads."""
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


@pytest.mark.parametrize("n_orb,n_el,rows,dtype", [(5, 5, 400, "c128"), (5, 4, 153, "c64"), (10, 6, 3, "c64"),
                                                   (9, 6, 2, "c128"), (4, 1, 2, "c128")])
def test_rows_match_single_calls(n_orb, n_el, rows, dtype):
    h, g = integrals(n_orb, 60 + n_orb)
    A, exs = prep.uccsd_ansatz(n_orb, n_el)
    T, det = prep.molecular_hamiltonian(h, g), (1 << n_el) - 1
    t = np.stack([amplitudes(len(exs), 500 + k, 0.15) for k in range(rows)])
    st, ref = qf.State(2 * n_orb, dtype), qf.State(2 * n_orb, dtype)
    st.energy_grad(det, A, t[0], T)
    qf.kernel_launches(True)
    e, gr = st.energy_grad_multi(det, A, t, T)
    assert qf.kernel_launches(True) == 2  # the grouped evaluation and the reset to |det>
    for k in {0, 1, rows // 2, rows - 1}:
        e1, g1 = ref.energy_grad(det, A, t[k], T)
        assert abs(e[k] - e1) < (1e-11 if dtype == "c128" else 2e-5)
        if dtype == "c128":
            assert np.abs(gr[k] - g1).max() < 1e-10
        else:
            assert np.linalg.norm(gr[k] - g1) <= 1e-4 * np.linalg.norm(g1)
    st.close(), ref.close()
