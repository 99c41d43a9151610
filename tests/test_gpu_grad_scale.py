"""The general path's complex64 gradient under Hamiltonians of any scale: products of psi, lambda
and the scale kept aside leave FP32's range long before either of them does."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()

from paper_2108_04413_gb300 import abi, qf  # noqa: E402


@pytest.mark.parametrize("factor", [1.0, 1e15, 1e24, 1e28, 1e-20, 1e-25])
def test_gradient_scales_with_the_hamiltonian(factor):
    n, m = 11, 58
    rng = np.random.default_rng(4)
    x = rng.integers(1, 1 << n, m) & rng.integers(1, 1 << n, m)
    z = rng.integers(0, 1 << n, m)
    # rotations by 0.8 put a factor of 0.717 each into the scale: 2^-28 before it is folded
    ansatz = abi.as_arots(x.astype(np.uint64), z.astype(np.uint64), np.full(m, 0.8), np.arange(m))
    hx = (rng.integers(0, 1 << n, 40) & rng.integers(0, 1 << n, 40)).astype(np.uint64)
    terms = abi.as_terms(hx, rng.integers(0, 1 << n, 40).astype(np.uint64), rng.normal(size=40))
    big = terms.copy()
    big["coeff"] *= factor
    st, ref = qf.State(n, "c64"), qf.State(n, "c128")
    e, g = st.energy_grad(5, ansatz, np.ones(m), big)
    e_ref, g_ref = ref.energy_grad(5, ansatz, np.ones(m), terms)
    assert abs(e / factor - e_ref) < 2e-5
    assert np.linalg.norm(g / factor - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    st.close(), ref.close()
