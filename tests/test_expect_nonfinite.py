"""Expectation passes on states with infinite, overflowing or undefined amplitudes give what the
per-group kernel gives (the allocation-free call): the infinity with its sign, or no number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()

from paper_2108_04413_gb300 import abi, qf  # noqa: E402


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e25, np.nan])
@pytest.mark.parametrize("terms_per_mask", [1, 6])
def test_same_as_the_group_kernel(dtype, value, terms_per_mask):
    n, masks = 16, 60
    # positive amplitudes and weights, so that only an infinite one is left to decide; 1e25
    # squared overflows complex64 products (the diagonal group)
    x = np.repeat(np.arange(masks, dtype=np.uint64) * np.uint64(37), terms_per_mask)
    z = np.tile(np.arange(terms_per_mask, dtype=np.uint64) << np.uint64(8), masks) & ~x
    coeff = np.tile(4.0 ** -np.arange(terms_per_mask), masks)  # the first outweighs the others
    terms = abi.as_terms(x, z, coeff)
    kind = np.complex64 if dtype == "c64" else np.complex128
    psi = np.full(1 << n, 2.0 ** -8, kind)
    psi[12345] = value
    st = qf.State(n, dtype)
    st.from_numpy(psi)
    got = st.expectation(terms)[0]
    dev = torch.from_numpy(psi).cuda()
    ref = qf.expectation_noalloc(dev.data_ptr(), n, dtype, torch.cuda.current_stream().cuda_stream, terms)[0]
    if np.isfinite(ref):  # complex128 holds 1e50
        assert abs(got - ref) <= 1e-12 * abs(ref)
    else:
        assert got == ref or (np.isnan(got) and np.isnan(ref))
    assert np.isfinite(ref) == (value == 1e25 and dtype == "c128")
    st.close()
