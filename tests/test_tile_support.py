"""Circuits on a determinant, whose first passes visit only the tiles the state has
reached: from few reached tiles to all of them, over several calls, and on amplitudes that
their owner overwrites in between; against a plain torch evaluation in complex128."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import __graft_entry__  # noqa: E402

__graft_entry__.build()

from paper_2108_04413_gb300 import abi, qf  # noqa: E402


def _reference(n, rots, psi):
    b = torch.arange(1 << n, device="cuda")
    for x, z, th in rots:
        s = torch.ones(1, dtype=torch.float64, device="cuda")
        for q in range(n):
            s = torch.cat([s, -s if (z >> q) & 1 else s])
        psi = math.cos(th) * psi - 1j * math.sin(th) * (1j ** bin(x & z).count("1")) * (s * psi)[b ^ x]
    return psi


def _rotations(n, count, rank, rng):
    """Random rotations whose X masks span `rank` dimensions (x = 0 and repeats among them)."""
    basis = [int(v) for v in rng.integers(1, 1 << n, rank)]
    basis[0] = 1 << (n - 1)
    out = []
    for _ in range(count):
        x = 0
        for v in rng.integers(0, rank, size=rng.integers(0, 3)):
            x ^= basis[v]
        if rng.integers(2):
            x &= int(rng.integers(0, 1 << n)) & int(rng.integers(0, 1 << n))
        out.append((x, int(rng.integers(0, 1 << n)), float(rng.uniform(-math.pi, math.pi))))
    return out


@pytest.mark.parametrize("n,rank", [(17, 3), (18, 1), (18, 4), (19, 6), (21, 5), (22, 12)])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
def test_circuit_on_a_determinant(n, rank, dtype, tol):
    rng = np.random.default_rng([n, rank])
    det = (1 << n) // 3
    kind = torch.complex128 if dtype == "c128" else torch.complex64
    buf = torch.empty(1 << n, dtype=kind, device="cuda")
    st = qf.State(n, dtype, buffer=buf)
    st.set_basis(det)
    ref = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    ref[det] = 1.0
    for count in (1, 7, 30):
        rots = _rotations(n, count, rank, rng)
        st.apply_circuit(abi.as_rots(*(list(c) for c in zip(*rots))))
        ref = _reference(n, rots, ref)
        st.apply_pauli_exp(1 << (n - 2), 5, 0.3)
        ref = _reference(n, [(1 << (n - 2), 5, 0.3)], ref)
    st.fold_scale()
    assert float((buf.to(torch.complex128) - ref).abs().max()) < tol


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
@pytest.mark.parametrize("where", ["all", "last"])
def test_amplitudes_written_by_their_owner(dtype, tol, where):
    n = 19
    rng = np.random.default_rng(5)
    kind = torch.complex128 if dtype == "c128" else torch.complex64
    buf = torch.empty(1 << n, dtype=kind, device="cuda")
    st = qf.State(n, dtype, buffer=buf)
    st.set_basis(0)
    if where == "all":
        buf.copy_(torch.full_like(buf, (1 << n) ** -0.5))
    else:
        buf.zero_()
        buf[-1] = 1.0
    ref = buf.to(torch.complex128, copy=True)
    rots = _rotations(n, 12, 3, rng)
    st.apply_circuit(abi.as_rots(*(list(c) for c in zip(*rots))))
    st.fold_scale()
    assert float((buf.to(torch.complex128) - _reference(n, rots, ref)).abs().max()) < tol
