"""Fused rotation passes on shared-memory tiles, forward and reverse, at the sizes where
the tile changes (10, 18-21 qubits) and with masks on the lowest and highest bits,
diagonal rotations, angles of both coefficient forms and a scale fold-back, against a
plain torch evaluation of the definitions in complex128."""
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


def _rotations(n, count, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 1 << n, count) & rng.integers(0, 1 << n, count) & rng.integers(0, 1 << n, count)
    z = rng.integers(0, 1 << n, count)
    x[::7] = 0
    for k, v in enumerate((1, 1 << (n - 1), 1 << 8, 1 << 9, (1 << 9) | 1, 1 << (n - 1) | 1 << 3, 3)):
        x[(5 * k + 1) % count] = v & ((1 << n) - 1)
    return x, z, rng.uniform(-math.pi, math.pi, count)


class Ref:
    def __init__(self, n):
        self.n, self.b = n, torch.arange(1 << n, device="cuda")

    def pauli(self, x, z, psi):
        s = torch.ones(1, dtype=torch.float64, device="cuda")
        for q in range(self.n):
            s = torch.cat([s, -s if (z >> q) & 1 else s])
        return 1j ** bin(x & z).count("1") * (s * psi)[self.b ^ x]

    def rotate(self, x, z, th, psi):
        return math.cos(th) * psi - 1j * math.sin(th) * self.pauli(x, z, psi)


@pytest.mark.parametrize("n,count", [(10, 40), (11, 60), (14, 60), (19, 40), (20, 60), (21, 60)])
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-12), ("c64", 2e-5)])
def test_circuit(n, count, dtype, tol):
    x, z, th = _rotations(n, count, n)
    det = (1 << n) // 3
    st, ref = qf.State(n, dtype), Ref(n)
    st.set_basis(det)
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[det] = 1.0
    for k in range(4):  # enough rotations to fold the kept scale in complex64
        st.apply_circuit(abi.as_rots(x, z, th + k))
        for a, b, t in zip(x.tolist(), z.tolist(), (th + k).tolist()):
            psi = ref.rotate(a, b, t, psi)
    assert np.abs(st.to_numpy() - psi.cpu().numpy()).max() < tol


@pytest.mark.parametrize("n,count", [(9, 20), (10, 30), (13, 40), (18, 30), (19, 30), (20, 30)])
@pytest.mark.parametrize("dtype,etol,gtol", [("c128", 1e-11, 1e-11), ("c64", 2e-5, 1e-4)])
def test_energy_gradient(n, count, dtype, etol, gtol):
    rng = np.random.default_rng(n)
    x, z, _ = _rotations(n, count, 50 + n)
    c, par, t = rng.normal(size=count), rng.integers(0, 7, count), rng.normal(size=7) * 0.4
    hx, hz, _ = _rotations(n, 25, 90 + n)
    hc = rng.normal(size=25) / 5
    det = (1 << n) // 5
    st, ref = qf.State(n, dtype), Ref(n)
    e, g = st.energy_grad(det, abi.as_arots(x, z, c, par), t, abi.as_terms(hx, hz, hc))
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[det] = 1.0
    rots = list(zip(x.tolist(), z.tolist(), c.tolist(), par.tolist()))
    for a, b, w, p in rots:
        psi = ref.rotate(a, b, w * t[p], psi)
    lam = sum(w * ref.pauli(a, b, psi) for a, b, w in zip(hx.tolist(), hz.tolist(), hc.tolist()))
    assert abs(e - torch.vdot(psi, lam).real.item()) < etol
    want = np.zeros(7)
    for a, b, w, p in reversed(rots):
        want[p] += 2 * w * torch.vdot(lam, ref.pauli(a, b, psi)).imag.item()
        psi, lam = ref.rotate(a, b, -w * t[p], psi), ref.rotate(a, b, -w * t[p], lam)
    assert np.linalg.norm(g - want) <= gtol * max(1.0, np.linalg.norm(want))
    e2, g2 = st.energy_grad(det, abi.as_arots(x, z, c, par), t, abi.as_terms(hx, hz, hc))
    assert e2 == e and np.array_equal(g, g2)  # fixed summation order
