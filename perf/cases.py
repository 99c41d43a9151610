"""The workloads this engine is timed on, through its public calls.

Seven kinds of work, each over the sizes the engine is used at (8 to 28 qubits,
complex128 and complex64):

* energy_grad: one VQE iteration, energy and gradient of a dUCCSD ansatz;
* multi: one serving batch, energies and gradients of many parameter vectors of one small molecule;
* pool: one ADAPT iteration, the gradients of an operator pool at the grown ansatz's state;
* circuit: a circuit of random Pauli exponentials on a determinant;
* expect: the expectation value of a random Hermitian Pauli sum in a given state;
* generic: energy and gradient of an ansatz of arbitrary Pauli exponentials (no particle-number symmetry);
* trotter: Trotterized time evolution of a determinant under a molecular Hamiltonian.

complex64 results are handed on in single precision: a gradient through the
torch.autograd wrapper with float32 parameters, batch results and expectation
values as float32.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_2108_04413_gb300 import abi, autograd, prep, qf


def listed():
    return [
        # the smallest molecule of the paper's dUCCSD timings (H4): launches and latency
        dict(name="energy_grad_8q_c128", what="energy_grad", orbitals=4, electrons=4, dtype="c128", sigma=0.1),
        # a VQE iteration of a medium molecule
        dict(name="energy_grad_16q_c128", what="energy_grad", orbitals=8, electrons=8, dtype="c128", sigma=0.1),
        # an open-shell cation, single precision, driven by a torch optimiser
        dict(name="energy_grad_20q_c64", what="energy_grad", orbitals=10, electrons=9, dtype="c64", sigma=0.05),
        # the headline evaluation: the largest system a VQE loop runs
        dict(name="energy_grad_24q_c128", what="energy_grad", orbitals=12, electrons=12, dtype="c128", sigma=0.05),
        # a group of requests of one small molecule taken together by the server
        dict(name="multi_14q_c64", what="multi", orbitals=7, electrons=7, rows=32, dtype="c64", sigma=0.1),
        # operator selection of ADAPT-VQE: a short grown ansatz, the whole dUCCSD pool
        dict(name="pool_20q_c128", what="pool", orbitals=10, electrons=10, operators=40, dtype="c128", sigma=0.1),
        # a general circuit on the largest register, FP64
        dict(name="circuit_28q_c128", what="circuit", qubits=28, rotations=100, dtype="c128"),
        # a longer general circuit, odd register, FP32
        dict(name="circuit_27q_c64", what="circuit", qubits=27, rotations=300, dtype="c64"),
        # energy of a general state under a general Pauli sum, odd register, FP64
        dict(name="expect_25q_c128", what="expect", qubits=25, terms=1500, dtype="c128"),
        # the same on the largest register, FP32
        dict(name="expect_28q_c64", what="expect", qubits=28, terms=500, dtype="c64"),
        # VQE with an ansatz outside the sector form (qubit-excitation / hardware-style), odd register
        dict(name="generic_17q_c128", what="generic", qubits=17, rotations=160, parameters=60, terms=400,
             dtype="c128"),
        # one time step of a quantum Krylov basis state
        dict(name="trotter_20q_c128", what="trotter", orbitals=10, electrons=10, steps=1, time=0.1, dtype="c128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["energy_grad", "energy_grad", "multi", "pool", "circuit", "circuit", "expect", "expect",
                       "generic", "trotter"])
    dtype = rng.choice(["c128", "c64"])
    if what == "energy_grad":
        no = rng.randint(4, 12)
        return dict(what=what, orbitals=no, electrons=rng.randint(max(2, no - 3), min(2 * no - 2, no + 2)),
                    dtype=dtype, sigma=rng.choice([0.05, 0.1]))
    if what == "multi":
        no = rng.randint(4, 8)
        return dict(what=what, orbitals=no, electrons=rng.randint(no - 2, no + 1), rows=_log_int(rng, 2, 64),
                    dtype=dtype, sigma=0.1)
    if what == "pool":
        no = rng.randint(5, 11)
        return dict(what=what, orbitals=no, electrons=rng.randint(no - 2, no + 1), operators=_log_int(rng, 2, 60),
                    dtype=dtype, sigma=0.1)
    if what == "circuit":
        n = rng.randint(10, 28)
        most = min(300, int((100 if dtype == "c128" else 250) * 2.0 ** (28 - n)))
        return dict(what=what, qubits=n, rotations=_log_int(rng, 4, most), dtype=dtype)
    if what == "expect":
        n = rng.randint(10, 28)
        most = min(2000, int((160 if dtype == "c128" else 500) * 2.0 ** (28 - n)))
        return dict(what=what, qubits=n, terms=_log_int(rng, 10, most), dtype=dtype)
    if what == "generic":
        n = rng.randint(8, 20)
        rots = _log_int(rng, 10, 200)
        return dict(what=what, qubits=n, rotations=rots, parameters=rng.randint(2, rots), terms=_log_int(rng, 10, 500),
                    dtype=dtype)
    no = rng.randint(4, 10)
    return dict(what=what, orbitals=no, electrons=rng.randint(no - 2, no + 2), steps=rng.randint(1, 2),
                time=rng.choice([0.05, 0.1, 0.2]), dtype=dtype)


# ---------------------------------------------------------------------------
# seeded inputs


def _integrals(no, rng):
    """Real symmetric h_pq and 8-fold symmetric (pq|rs), the shape of molecular integrals in a local basis."""
    h = rng.normal(0.0, 0.1, size=(no, no))
    h = np.triu(h, 1) + np.triu(h, 1).T + np.diag(rng.uniform(-2.0, 0.0, size=no))
    g = rng.normal(0.0, 0.05, size=(no,) * 4)
    d = np.exp(-np.abs(np.arange(no)[:, None] - np.arange(no)[None, :]).astype(float))
    pair = np.arange(no * no).reshape(no, no)
    pair = np.minimum(pair, pair.T)  # one index per unordered pair
    a, b = pair[:, :, None, None], pair[None, None, :, :]
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    g = g.reshape(no * no, no * no)[lo, hi]
    return h, g * d[:, :, None, None] * d[None, None, :, :]


def _masks(n, count, rng):
    """Random Pauli strings: weight 2 to 8, letters uniform in X, Y, Z."""
    x, z = np.zeros(count, np.uint64), np.zeros(count, np.uint64)
    for k in range(count):
        w = int(rng.integers(2, min(8, n) + 1))
        for q, letter in zip(rng.choice(n, size=w, replace=False), rng.integers(0, 3, size=w)):
            x[k] |= np.uint64((letter != 2) << int(q))
            z[k] |= np.uint64((letter != 0) << int(q))
    return x, z


@functools.lru_cache(maxsize=4)
def _uccsd(no, ne):
    return prep.uccsd_ansatz(no, ne)


def _subset(ansatz, keep):
    """The rotations of the operators `keep`, in that order, with parameters 0, 1, ..."""
    rows = [ansatz[ansatz["param"] == mu].copy() for mu in keep]
    for k, r in enumerate(rows):
        r["param"] = k
    return np.concatenate(rows)


def _draws(case, seed):
    """Every random number of a case (used by prepare and by exact)."""
    rng = np.random.default_rng([2108, int(seed)])
    what = case["what"]
    d = {}
    if what in ("energy_grad", "multi", "pool", "trotter"):
        d["h"], d["g"] = _integrals(case["orbitals"], rng)
        d["det"] = (1 << case["electrons"]) - 1
    if what in ("energy_grad", "multi", "pool"):
        npar = len(_excitations(case["orbitals"], case["electrons"]))
        if what == "pool":
            d["keep"] = rng.permutation(npar)[:case["operators"]]
            npar = len(d["keep"])
        shape = (case["rows"], npar) if what == "multi" else (npar,)
        d["t"] = rng.normal(0.0, case["sigma"], size=shape)
        if case["dtype"] == "c64" and what == "energy_grad":
            d["t"] = d["t"].astype(np.float32)
    if what in ("circuit", "generic"):
        n, m = case["qubits"], case["rotations"]
        d["x"], d["z"] = _masks(n, m, rng)
        d["det"] = int(rng.integers(0, 1 << n))
        d["theta"] = rng.uniform(-math.pi, math.pi, size=m)
        if what == "generic":
            d["coeff"] = rng.normal(0.0, 1.0, size=m)
            d["param"] = np.concatenate([np.arange(case["parameters"]),
                                         rng.integers(0, case["parameters"], size=m - case["parameters"])])
            d["t"] = rng.normal(0.0, 0.3, size=case["parameters"])
            if case["dtype"] == "c64":
                d["t"] = d["t"].astype(np.float32)
    if what in ("expect", "generic"):
        n, m = case["qubits"], case["terms"]
        d["hx"], d["hz"] = _masks(n, m, rng)
        d["hc"] = rng.normal(0.0, 1.0, size=m) / math.sqrt(m)
    if what == "expect":
        d["tilt"], d["turn"] = rng.uniform(0.2, 1.3, size=case["qubits"]), rng.uniform(-1.5, 1.5, size=case["qubits"])
        d["noise"] = int(rng.integers(1 << 31))
    return d


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _state_vector(d, n, dtype):
    """A normalised state: a product of single-qubit states with 5 % of noise on every amplitude."""
    dev = _device()
    psi = torch.ones(1, dtype=torch.complex64, device=dev)
    for q in range(n):  # qubit q is bit q
        a, b = d["tilt"][q], d["turn"][q]
        psi = torch.cat([psi * math.cos(a), psi * (math.sin(a) * complex(math.cos(b), math.sin(b)))])
    gen = torch.Generator(device=dev)
    gen.manual_seed(d["noise"])
    psi *= 1.0 + 0.05 * torch.randn(1 << n, generator=gen, device=dev)
    psi = psi.to(dtype)
    return psi.div_(float(torch.linalg.vector_norm(psi)))


# ---------------------------------------------------------------------------


def prepare(case, seed):
    what, dtype = case["what"], case["dtype"]
    d = _draws(case, seed)
    s = dict(case)
    if what in ("energy_grad", "multi", "pool", "trotter"):
        n = 2 * case["orbitals"]
        s["terms"] = prep.molecular_hamiltonian(d["h"], d["g"])
    else:
        n = case["qubits"]
    if what in ("circuit", "trotter"):  # the program owns the amplitudes
        s["psi"] = torch.empty(1 << n, dtype=torch.complex128 if dtype == "c128" else torch.complex64, device="cuda")
        s["state"] = qf.State(n, dtype, buffer=s["psi"])
    else:
        s["state"] = qf.State(n, dtype)
    if what in ("energy_grad", "multi", "pool"):
        ansatz, _ = _uccsd(case["orbitals"], case["electrons"])
        s["ansatz"] = ansatz
        if what == "pool":
            s["ansatz"], s["pool"], s["n_pool"] = _subset(ansatz, d["keep"]), ansatz, int(ansatz["param"].max()) + 1
    if what == "circuit":
        s["rots"] = abi.as_rots(d["x"], d["z"], d["theta"])
    if what == "generic":
        s["ansatz"] = abi.as_arots(d["x"], d["z"], d["coeff"], d["param"])
    if what in ("expect", "generic"):
        s["terms"] = abi.as_terms(d["hx"], d["hz"], d["hc"])
    if what == "expect":
        s["state"].from_numpy(_state_vector(d, n, torch.complex128 if dtype == "c128" else torch.complex64)
                              .cpu().numpy())
    s["det"] = d.get("det")
    if "t" in d:
        s["t"] = d["t"]
        if dtype == "c64" and what in ("energy_grad", "generic"):
            s["t"] = torch.tensor(d["t"], dtype=torch.float32, device="cuda", requires_grad=True)
    return s


def run(s):
    what, single, st = s["what"], s["dtype"] == "c64", s["state"]
    if what in ("energy_grad", "generic"):
        if single:
            t = s["t"]
            t.grad = None
            e = autograd.energy(t, st, s["det"], s["ansatz"], s["terms"])
            e.backward()
            return {"energy": e.detach(), "grad": t.grad}
        e, g = st.energy_grad(s["det"], s["ansatz"], s["t"], s["terms"])
        return {"energy": np.float64(e), "grad": g}
    if what == "multi":
        e, g = st.energy_grad_multi(s["det"], s["ansatz"], s["t"], s["terms"])
        return {"energy": e.astype(np.float32), "grad": g.astype(np.float32)} if single else {"energy": e, "grad": g}
    if what == "pool":
        e, g = st.pool_gradients(s["det"], s["ansatz"], s["t"], s["terms"], s["pool"], s["n_pool"])
        kind = np.float32 if single else np.float64
        return {"energy": kind(e), "grad": g.astype(kind)}
    if what == "circuit":
        st.set_basis(s["det"])
        st.apply_circuit(s["rots"])
        st.fold_scale()
        return s["psi"]
    if what == "trotter":
        st.set_basis(s["det"])
        st.trotter(s["terms"], s["time"], s["steps"])
        st.fold_scale()
        return s["psi"]
    re, _ = st.expectation(s["terms"])
    return np.float32(re) if single else np.float64(re)


def work(case):
    what = case["what"]
    size = 16 if case["dtype"] == "c128" else 8
    if what in ("energy_grad", "multi", "pool"):
        no, ne = case["orbitals"], case["electrons"]
        na, nb = (ne + 1) // 2, ne // 2
        members = math.comb(no, na) * math.comb(no, nb)
        items = 0  # (determinant pair, excitation) rotations of one sweep
        exs = _excitations(no, ne)
        for occ, vir in exs:
            ka, kb = sum(p % 2 == 0 for p in occ), sum(p % 2 == 1 for p in occ)
            items += math.comb(no - 2 * ka, na - ka) * math.comb(no - 2 * kb, nb - kb)
        sa, sb = na * (no - na), nb * (no - nb)
        daa, dbb = (math.comb(na, 2) * math.comb(no - na, 2), math.comb(nb, 2) * math.comb(no - nb, 2))
        links = 1 + sa + sb + daa + dbb + sa * sb  # determinants H connects to one determinant
        hpsi = 2 * links * members
        if what == "pool":
            return {"bytes": members * size + 8 * len(exs), "flops": hpsi + 6 * items}
        one = {"bytes": members * size + 16 * len(exs), "flops": hpsi + (8 + 14) * items}
        rows = case.get("rows", 1)
        return {k: v * rows for k, v in one.items()}
    if what == "trotter":
        n = 2 * case["orbitals"]
        no = case["orbitals"]
        # one 2x2 real rotation of every amplitude per flip pattern of the Hamiltonian (its Pauli strings commute)
        groups = 1 + 2 * math.comb(no, 2) + 2 * math.comb(no, 4) + math.comb(no, 2) ** 2
        return {"bytes": size << n, "flops": case["steps"] * groups * (4 << n)}
    n = case["qubits"]
    if what == "circuit":
        return {"bytes": size << n, "flops": case["rotations"] * (4 << n)}
    if what == "expect":
        return {"bytes": size << n, "flops": case["terms"] * (2 << n)}
    return {"bytes": size << n, "flops": (3 * case["rotations"] + 2 * case["terms"]) * (4 << n)}


# ---------------------------------------------------------------------------
# the same results from the definitions, in 64 bits


def _excitations(no, ne):
    """Spin-conserving singles and doubles of the lowest-ne determinant, by the excited determinant's value."""
    occ, vir = range(ne), range(ne, 2 * no)
    exs = [((i,), (a,)) for i in occ for a in vir if i % 2 == a % 2]
    exs += [(o, v) for o in itertools.combinations(occ, 2) for v in itertools.combinations(vir, 2)
            if sum(p % 2 for p in o) == sum(p % 2 for p in v)]
    return sorted(exs, key=lambda e: sum(1 << a for a in e[1]) - sum(1 << i for i in e[0]))


class _Sector:
    """The determinants with the reference's numbers of alpha (even) and beta (odd) electrons."""

    def __init__(self, no, ne, dev):
        self.no, self.n, self.dev = no, 2 * no, dev
        alpha = [sum(1 << 2 * p for p in c) for c in itertools.combinations(range(no), (ne + 1) // 2)]
        beta = [sum(2 << 2 * p for p in c) for c in itertools.combinations(range(no), ne // 2)]
        dets = torch.tensor(alpha, device=dev)[:, None] + torch.tensor(beta, device=dev)[None, :]
        self.dets = dets.reshape(-1)
        self.pos = torch.full((1 << self.n,), -1, dtype=torch.int64, device=dev)
        self.pos[self.dets] = torch.arange(len(self.dets), device=dev)

    def _parity(self, d, p):
        """(-1)^(electrons in orbitals below p)."""
        v = d & ((1 << p) - 1)
        for k in (16, 8, 4, 2, 1):
            v = v ^ (v >> k)
        return 1.0 - 2.0 * (v & 1).double()

    def link(self, create, remove):
        """Indices (i0, i1) and signs with a+_create... a_remove... |i0> = sign |i1>, rightmost operator first."""
        d = self.dets
        has, empty = sum(1 << p for p in remove), sum(1 << p for p in create if p not in remove)
        i0 = torch.nonzero(((d & has) == has) & ((d & empty) == 0)).reshape(-1)
        d = d[i0]
        sign = torch.ones(len(d), dtype=torch.float64, device=self.dev)
        for p in list(reversed(list(create) + list(remove))):
            sign = sign * self._parity(d, p)
            d = d ^ (1 << p)
        return i0, self.pos[d], sign

    def tau(self, ex):
        occ, vir = ex
        return self.link(list(vir), list(reversed(occ)))

    def hamiltonian(self, h, g, psi):
        """H psi from E_pq = sum_s a+_ps a_qs: sum (h_pq - sum_r (pr|rq)/2) E_pq + sum (pq|rs)/2 E_pq E_rs."""
        no, dev = self.no, self.dev
        rows, m = psi.shape
        h = torch.tensor(h - 0.5 * np.einsum("prrq->pq", g), device=dev)
        g = torch.tensor(0.5 * g.reshape(no * no, no * no), device=dev)
        links = [[self.link([2 * p + s], [2 * q + s]) for s in (0, 1)] for p in range(no) for q in range(no)]
        out = torch.zeros_like(psi)
        for r in range(rows):
            e = torch.zeros((no * no, m), dtype=torch.float64, device=dev)
            for k, both in enumerate(links):
                for i0, i1, sign in both:
                    e[k].index_add_(0, i1, sign * psi[r, i0])
            w = g @ e
            w += h.reshape(-1, 1) * psi[r]
            for k, both in enumerate(links):
                for i0, i1, sign in both:
                    out[r].index_add_(0, i1, sign * w[k, i0])
        return out

    def factor(self, v, link, t):
        """exp(t (tau - tau+)) v, t one angle per row of v."""
        i0, i1, sign = link
        c, s = torch.cos(t)[:, None], torch.sin(t)[:, None] * sign
        a, b = v[:, i0], v[:, i1]
        v[:, i0], v[:, i1] = c * a - s * b, c * b + s * a

    def overlap(self, lam, psi, link):
        i0, i1, sign = link
        return 2.0 * (sign * (lam[:, i1] * psi[:, i0] - lam[:, i0] * psi[:, i1])).sum(1)


def _exact_ucc(case, d):
    dev = _device()
    no, ne = case["orbitals"], case["electrons"]
    sec = _Sector(no, ne, dev)
    exs = _excitations(no, ne)
    t = torch.tensor(np.atleast_2d(d["t"]), dtype=torch.float64, device=dev)
    ops = [exs[k] for k in d["keep"]] if case["what"] == "pool" else exs
    psi = torch.zeros((len(t), len(sec.dets)), dtype=torch.float64, device=dev)
    psi[:, sec.pos[d["det"]]] = 1.0
    for k, ex in enumerate(ops):
        sec.factor(psi, sec.tau(ex), t[:, k])
    lam = sec.hamiltonian(d["h"], d["g"], psi)
    e = (psi * lam).sum(1)
    if case["what"] == "pool":
        grad = torch.stack([sec.overlap(lam, psi, sec.tau(ex)) for ex in exs], 1)
    else:
        grad = torch.zeros_like(t)
        for k in reversed(range(len(ops))):
            link = sec.tau(ops[k])
            grad[:, k] = sec.overlap(lam, psi, link)
            sec.factor(psi, link, -t[:, k])
            sec.factor(lam, link, -t[:, k])
    if case["what"] != "multi":
        e, grad = e[0], grad[0]
    return {"energy": e, "grad": grad}


class _Register:
    """The whole register of n qubits: P|b> = i^popc(x&z) (-1)^popc(z&b) |b^x>."""

    def __init__(self, n, dev):
        self.n, self.dev = n, dev
        self.b = torch.arange(1 << n, device=dev)

    def sign(self, z):
        s = torch.ones(1, dtype=torch.int8, device=self.dev)
        for q in range(self.n):
            s = torch.cat([s, -s if (z >> q) & 1 else s])
        return s

    def pauli(self, x, z, psi):
        """P psi."""
        flip = 1 - 2 * (bin(x & z).count("1") & 1)  # (-1)^popc(z & x): the sign at b^x against that at b
        v = psi[self.b ^ x] if x else psi.clone()
        v *= self.sign(z)
        return v.mul_(flip * (1, 1j, -1, -1j)[bin(x & z).count("1") & 3])

    def rotate(self, x, z, theta, psi):
        v = self.pauli(x, z, psi)
        psi *= math.cos(theta)
        psi -= v.mul_(1j * math.sin(theta))

    def basis(self, det):
        psi = torch.zeros(1 << self.n, dtype=torch.complex128, device=self.dev)
        psi[det] = 1.0
        return psi


def _popcount(a):
    return np.bitwise_count(a.astype(np.uint64)).astype(np.int64)


def _strings(h, g):
    """The Pauli strings (x, z, c) of the molecular Hamiltonian, ordered by (x, z): products of the
    Jordan-Wigner images of E_pq = sum_s a+_ps a_qs, each string kept as c X^x Z^z (Z acts first)."""
    no = len(h)
    idx, xs, zs, cs = [], [], [], []
    for p, q, s in itertools.product(range(no), range(no), range(2)):
        a, b = 2 * p + s, 2 * q + s
        for u, v in itertools.product((0, 1), (0, 1)):  # a+ = X Z..(1 + Z)/2, a = X Z..(1 - Z)/2
            z1, z2 = (1 << a) - 1 | u << a, (1 << b) - 1 | v << b
            idx.append(p * no + q)
            xs.append(1 << a ^ 1 << b)
            zs.append(z1 ^ z2)
            cs.append((-0.25 if v else 0.25) * (-1) ** (z1 >> b & 1))
    idx, xs, zs, cs = np.array(idx), np.array(xs), np.array(zs), np.array(cs, float)
    one = (h - 0.5 * np.einsum("prrq->pq", g)).reshape(-1)[idx] * cs
    two = 0.5 * g.reshape(no * no, no * no)[idx[:, None], idx[None, :]] * cs[:, None] * cs[None, :]
    two *= 1 - 2 * (_popcount(zs[:, None] & xs[None, :]) & 1)
    x = np.concatenate([xs, (xs[:, None] ^ xs[None, :]).reshape(-1)])
    z = np.concatenate([zs, (zs[:, None] ^ zs[None, :]).reshape(-1)])
    key, at = np.unique(x << 32 | z, return_inverse=True)
    c = np.bincount(at.reshape(-1), np.concatenate([one, two.reshape(-1)]))
    x, z = key >> 32, key & 0xFFFFFFFF
    c = c * np.array([1, 0, -1, 0])[_popcount(x & z) & 3]  # X^x Z^z = (-i)^popc(x&z) P; odd powers cancel
    return [(int(x[k]), int(z[k]), float(c[k])) for k in np.nonzero(np.abs(c) > 1e-14)[0]]


def exact(case, seed):
    what = case["what"]
    d = _draws(case, seed)
    if what in ("energy_grad", "multi", "pool"):
        return _exact_ucc(case, d)
    dev = _device()
    if what == "trotter":
        reg = _Register(2 * case["orbitals"], dev)
        psi = reg.basis(d["det"])
        strings = _strings(d["h"], d["g"])
        for _ in range(case["steps"]):
            for x, z, c in strings:
                reg.rotate(x, z, c * case["time"] / case["steps"], psi)
        return psi
    reg = _Register(case["qubits"], dev)
    if what == "circuit":
        psi = reg.basis(d["det"])
        for x, z, th in zip(d["x"].tolist(), d["z"].tolist(), d["theta"].tolist()):
            reg.rotate(x, z, th, psi)
        return psi
    terms = list(zip(d["hx"].tolist(), d["hz"].tolist(), d["hc"].tolist()))
    if what == "expect":
        kind = torch.complex128 if case["dtype"] == "c128" else torch.complex64
        psi = _state_vector(d, case["qubits"], kind).to(torch.complex128)
        total = 0.0
        for x, group in itertools.groupby(sorted(terms), key=lambda term: term[0]):
            w = psi[reg.b ^ x].conj_physical_().mul_(psi)  # conj(psi[b^x]) psi[b]
            for _, z, c in group:
                v = w  # sum_b (-1)^popc(z & b) w[b], one qubit at a time
                for q in reversed(range(case["qubits"])):
                    v = v.view(2, -1)
                    v = v[0] - v[1] if (z >> q) & 1 else v[0] + v[1]
                phase = (1, 1j, -1, -1j)[bin(x & z).count("1") & 3]
                total += c * (phase * complex(v.item())).real
        return torch.tensor(total, dtype=torch.float64)
    # generic
    t = d["t"].astype(np.float64)
    rots = list(zip(d["x"].tolist(), d["z"].tolist(), d["coeff"].tolist(), d["param"].tolist()))
    psi = reg.basis(d["det"])
    for x, z, c, p in rots:
        reg.rotate(x, z, c * t[p], psi)
    lam = torch.zeros_like(psi)
    for x, z, c in terms:
        lam += c * reg.pauli(x, z, psi)
    e = torch.vdot(psi, lam).real
    grad = torch.zeros(len(t), dtype=torch.float64, device=dev)
    for x, z, c, p in reversed(rots):
        grad[p] += 2.0 * c * torch.vdot(lam, reg.pauli(x, z, psi)).imag
        reg.rotate(x, z, -c * t[p], psi)
        reg.rotate(x, z, -c * t[p], lam)
    return {"energy": e, "grad": grad}
