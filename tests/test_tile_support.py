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


@pytest.mark.parametrize("orbitals,electrons,steps,count", [(4, 3, 2, 12), (5, 5, 1, 12), (5, 4, 1, 999),
                                                            (7, 6, 1, 999), (9, 7, 2, 12), (9, 8, 1, 150)])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
def test_trotter_blocks(orbitals, electrons, steps, count, dtype, tol):
    """Composite blocks of one to three row pairs, real and imaginary links, before and
    after the state has reached every pattern."""
    from paper_2108_04413_gb300 import prep

    n = 2 * orbitals
    rng = np.random.default_rng(orbitals)
    h = rng.normal(size=(orbitals, orbitals))
    g = rng.normal(size=(orbitals,) * 4)
    g = g + g.transpose(1, 0, 2, 3)
    g = g + g.transpose(0, 1, 3, 2)
    g = g + g.transpose(2, 3, 0, 1)
    terms = prep.molecular_hamiltonian(h + h.T, 0.2 * g)
    xs = np.unique(terms["x"])
    same = [x for x in xs if bin(int(x)).count("1") == 4 and bin(int(x) & 0x155555).count("1") in (0, 4)]
    few = rng.choice(xs, size=min(len(xs), 12), replace=False)
    keep = list(few if count == 12 else xs[:count]) + same[:3]
    terms = terms[np.isin(terms["x"], keep)]
    kind = torch.complex128 if dtype == "c128" else torch.complex64
    buf = torch.empty(1 << n, dtype=kind, device="cuda")
    st = qf.State(n, dtype, buffer=buf)
    det = (1 << electrons) - 1
    ansatz, _ = prep.uccsd_ansatz(orbitals, electrons)
    real = prep.bind_thetas(ansatz, rng.normal(0, 0.3, size=int(ansatz["param"].max()) + 1))[:40]
    for start in ("determinant", "turned", "written"):
        st.set_basis(det)
        ref = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
        ref[det] = 1.0
        if start == "turned":  # excitations' real blocks on a complex state
            st.apply_pauli_exp(3, 1, 0.4)
            st.apply_pauli_exp(0, 2, 0.4)
            ref = _reference(n, [(3, 1, 0.4), (0, 2, 0.4)], ref)
            st.apply_circuit(real)
            ref = _reference(n, list(zip(real["x"].tolist(), real["z"].tolist(), real["theta"].tolist())), ref)
        if start == "written":
            st.from_numpy(np.full(1 << n, 2.0 ** (-n / 2), dtype=np.complex128 if dtype == "c128" else np.complex64))
            ref = torch.full_like(ref, 2.0 ** (-n / 2))
        st.trotter(terms, 0.3, steps)
        st.fold_scale()
        for _ in range(steps):
            ref = _reference(n, [(int(t["x"]), int(t["z"]), float(t["coeff"]) * 0.3 / steps) for t in terms], ref)
        assert float((buf.to(torch.complex128) - ref).abs().max()) < tol


@pytest.mark.parametrize("n,count", [(1, 30), (6, 24), (13, 40), (18, 300), (19, 23)])
@pytest.mark.parametrize("parity", [0, 1])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
def test_runs_of_one_x_mask(n, count, parity, dtype, tol):
    """Commuting strings of one X mask, all with an even or all with an odd number of Y, and
    a diagonal run, on a determinant, on a spread state and on one written by its owner."""
    rng = np.random.default_rng([n, count, parity])
    kind = torch.complex128 if dtype == "c128" else torch.complex64
    buf = torch.empty(1 << n, dtype=kind, device="cuda")
    st = qf.State(n, dtype, buffer=buf)
    det = (1 << n) // 3
    st.set_basis(det)
    ref = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    ref[det] = 1.0
    for step in range(4):
        x = int(rng.integers(1, 1 << n)) if step != 2 else 0
        rots = []
        while len(rots) < count:
            z = int(rng.integers(0, 1 << n))
            if x == 0 or bin(x & z).count("1") % 2 == parity:
                rots.append((x, z, float(rng.uniform(-math.pi, math.pi))))
        if step == 3:
            st.fold_scale()
            buf.copy_(torch.full_like(buf, 2.0 ** (-n / 2)))
            ref = buf.to(torch.complex128, copy=True)
        st.apply_circuit(abi.as_rots(*(list(c) for c in zip(*rots))))
        ref = _reference(n, rots, ref)
    st.fold_scale()
    assert float((buf.to(torch.complex128) - ref).abs().max()) < tol
