"""Grouped requests whose H|psi> overflows give gradients that say so, as qf_energy_grad does."""
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


@pytest.mark.parametrize("dtype,factor,finite", [("c64", 1e30, True), ("c64", 1e39, False), ("c64", 1e300, False),
                                                 ("c128", 1e39, True), ("c128", 1e300, True)])
def test_overflowing_hamiltonian(dtype, factor, finite):
    h, g = integrals(5, 1)
    A, exs = prep.uccsd_ansatz(5, 5)
    T = prep.molecular_hamiltonian(h, g)
    t = np.stack([amplitudes(len(exs), k, 0.1) for k in range(3)])
    st, one = qf.State(10, dtype), qf.State(10, dtype)
    _, ref = one.energy_grad_multi(31, A, t, T)
    big = T.copy()
    big["coeff"] *= factor
    st.energy_grad(31, A, t[0], big)
    qf.kernel_launches(True)
    _, gr = st.energy_grad_multi(31, A, t, big)
    assert qf.kernel_launches(True) == 2  # grouped
    if finite:
        assert np.abs(gr / factor - ref).max() < (1e-10 if dtype == "c128" else 1e-4)
    else:
        assert not np.isfinite(gr).any()
    st.close(), one.close()
