"""Workloads of the state-vector emulator, each one pass through the public
entry points of ``paper_1604_06460_gb300.qe``.

A case names a kind of work and its sizes:

- ``circuit``: a random circuit (layers of a Haar-random U(2) on every qubit,
  then CNOTs on disjoint random pairs) applied gate by gate (``max_k`` 1) or
  fused to the library's default width (``max_k`` 0);
- ``qft``: the emulated quantum Fourier transform of a contiguous register;
- ``add``: the emulated addition of a classical constant to a register;
- ``muldiv``: the emulated multiplication and division of three registers;
- ``observe``: a Hamiltonian's energy, a marginal distribution and samples;
- ``batch``: many small ansatz circuits of mixed size, each returning an energy;
- ``qpe``: phase estimation by emulation with a dense unitary.

``prepare`` draws everything from the seed (the state by torch, in place in the
buffer that the state borrows), ``run`` is one pass, ``exact`` the same result
from plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1604_06460_gb300 import qe

LAYERS = 8       # layers of a batch's ansatz circuits
HX = 0.7         # transverse field of the Ising chain


def listed():
    return [
        # a ten-qubit circuit: what a user tries first, and what variational
        # loops call thousands of times; launches and host work decide
        {"name": "circuit_small_c128", "kind": "circuit", "n": 10, "depth": 3, "max_k": 0, "dtype": "c128", "arith": "fp64"},
        # gate-by-gate simulation without fusion (20 qubits, 10 layers)
        {"name": "gates_n20_c128", "kind": "circuit", "n": 20, "depth": 10, "max_k": 1, "dtype": "c128", "arith": "fp64"},
        # the fused circuit in the default arithmetic, at a size well beyond the caches
        {"name": "circuit_n28_c128", "kind": "circuit", "n": 28, "depth": 6, "max_k": 0, "dtype": "c128", "arith": "fp64"},
        # the same circuit family on a single-precision state
        {"name": "circuit_n29_c64", "kind": "circuit", "n": 29, "depth": 6, "max_k": 0, "dtype": "c64", "arith": "fp64"},
        # the Fourier transform of a whole 30-qubit state
        {"name": "qft_n30_c128", "kind": "qft", "n": 30, "lo": 0, "m": 30, "inverse": False, "dtype": "c128", "arith": "fp64"},
        # an inverse transform of an odd register in the middle of a state,
        # as phase estimation ends with
        {"name": "qft_reg_n27_c128", "kind": "qft", "n": 27, "lo": 5, "m": 17, "inverse": True, "dtype": "c128", "arith": "fp64"},
        # the whole-state transform in single precision, at an odd size
        {"name": "qft_n27_c64", "kind": "qft", "n": 27, "lo": 0, "m": 27, "inverse": False, "dtype": "c64", "arith": "fp64"},
        # a classical constant added to a 16-qubit register
        {"name": "add_n29_c128", "kind": "add", "n": 29, "lo": 0, "m": 16, "stride": 1, "dtype": "c128", "arith": "fp64"},
        # reversible multiplication and division of nine-qubit registers
        {"name": "muldiv_n28_c128", "kind": "muldiv", "n": 28, "N": 9, "lo": 0, "dtype": "c128", "arith": "fp64"},
        # what is read out at a circuit's end: the Ising energy, a marginal, samples
        {"name": "observe_n28_c128", "kind": "observe", "n": 28, "ham": "ising", "m": 3, "shots": 4096, "dtype": "c128", "arith": "fp64"},
        # a parameter sweep: circuits of 10 to 22 qubits in one launch
        {"name": "batch_c128", "kind": "batch", "count": 512, "nlo": 10, "nhi": 22, "dtype": "c128", "arith": "df64"},
        # phase estimation of a Trotter step on 10 qubits with 8 result bits
        {"name": "qpe_n18_c128", "kind": "qpe", "nsys": 10, "b": 8, "dtype": "c128", "arith": "fp64"},
    ]


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "qft", "qft", "add", "muldiv", "observe", "batch", "qpe"])
    dtype, arith = rng.choice([("c128", "fp64"), ("c128", "fp64"), ("c64", "fp64"), ("c128", "df64")])
    case = {"kind": kind}
    if kind == "circuit":
        by_gate = rng.random() < 0.3
        n = rng.randint(10, 23) if by_gate else rng.randint(10, 28)
        case.update(n=n, depth=rng.randint(2, 6), max_k=1 if by_gate else 0)
    elif kind == "qft":
        n = rng.randint(10, 28)
        m = n if rng.random() < 0.4 else rng.randint(1, n)
        case.update(n=n, lo=rng.randint(0, n - m), m=m, inverse=rng.random() < 0.5)
    elif kind == "add":
        n = rng.randint(10, 29)
        stride = 2 if rng.random() < 0.2 else 1
        m = rng.randint(1, min(n // stride, 18))
        case.update(n=n, lo=rng.randint(0, n - stride * (m - 1) - 1), m=m, stride=stride)
    elif kind == "muldiv":
        n = rng.randint(12, 27)
        N = rng.randint(2, min(n // 3, 9))
        case.update(n=n, N=N, lo=rng.randint(0, n - 3 * N))
    elif kind == "observe":
        n = rng.randint(10, 28)
        case.update(n=n, ham=rng.choice(["ising", "heisenberg"]), m=rng.randint(1, min(n, 8)), shots=rng.choice([1, 100, 1000, 4096, 10000]))
    elif kind == "batch":
        nlo = rng.randint(4, 14)
        nhi = rng.randint(nlo, 22)
        if dtype == "c128" and rng.random() < 0.5:
            arith = "df64"       # the batch's default
        # at most the listed batch's amplitudes, a quarter of them in FP64
        mean = (2 ** (nhi + 1) - 2 ** nlo) / (nhi + 1 - nlo)
        most = 3.3e8 / mean / (4 if (dtype, arith) == ("c128", "fp64") else 1)
        case.update(count=max(1, int(min(2 ** rng.uniform(4, 9), most))), nlo=nlo, nhi=nhi)
    else:
        dtype = "c128"
        arith = "fp64" if arith == "df64" and rng.random() < 0.5 else arith
        case.update(nsys=rng.randint(3, 10), b=rng.randint(3, 8))
    case.update(dtype=dtype, arith=arith)
    return case


# --------------------------------------------------------------- inputs
def _real(case):
    return torch.float64 if case["dtype"] == "c128" else torch.float32


def _amplitudes(n, seed, real):
    """A normalised complex Gaussian state, interleaved."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(2 << n, generator=g, device="cuda", dtype=torch.float64 if real == torch.float64 else torch.float32)
    scale = 1.0 / math.sqrt(float(torch.dot(x, x)) if n <= 24 else float(sum(torch.dot(c, c).double() for c in x.split(1 << 25))))
    return x.mul_(scale)


def _haar(rng):
    z = rng.standard_normal((2, 2)) + 1j * rng.standard_normal((2, 2))
    q, r = np.linalg.qr(z)
    d = np.diag(r)
    return q * (d / np.abs(d))[None, :]


CNOT = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], dtype=np.complex128)


def _circuit(n, depth, seed):
    """(qubits, matrix) of every gate; a CNOT's qubits are (target, control)."""
    rng = np.random.default_rng(seed)
    gates = []
    for _ in range(depth):
        gates += [((q,), _haar(rng)) for q in range(n)]
        p = rng.permutation(n)
        gates += [((int(p[2 * j + 1]), int(p[2 * j])), CNOT) for j in range(n // 2)]
    return gates


def _trotter(n, seed):
    """One Trotter step of the transverse-field Ising chain with seeded angles."""
    rng = np.random.default_rng(seed)
    gates = []
    for i in range(n - 1):
        t = rng.uniform(0.1, 0.4)
        rz = np.diag([np.exp(-0.5j * t), np.exp(0.5j * t)])
        gates += [((i + 1, i), CNOT), ((i + 1,), rz), ((i + 1, i), CNOT)]
    for q in range(n):
        t = rng.uniform(0.05, 0.3)
        gates.append(((q,), np.array([[np.cos(t), -1j * np.sin(t)], [-1j * np.sin(t), np.cos(t)]])))
    return gates


def _constant(case, seed):
    return int(np.random.default_rng(seed).integers(1, 1 << case["m"])) if case["m"] > 1 else 1


def _register(case):
    return [case["lo"] + case["stride"] * j for j in range(case["m"])]


def _registers(case):
    """a, b, c with c in the low qubits and a on top, as the paper writes a b c."""
    N, lo = case["N"], case["lo"]
    return [list(range(lo + k * N, lo + (k + 1) * N)) for k in (2, 1, 0)]


def _hamiltonian(case):
    """Pauli masks (x, z) and coefficients of a nearest-neighbour chain."""
    n, xm, zm, cf = case["n"], [], [], []
    for i in range(n - 1):
        pair = (1 << i) | (1 << (i + 1))
        for x, z, c in ([(0, pair, 1.0)] if case["ham"] == "ising" else [(pair, 0, 1.0), (pair, pair, 0.9), (0, pair, 1.1)]):
            xm.append(x)
            zm.append(z)
            cf.append(c)
    for i in range(n):
        x, z, c = (1 << i, 0, HX) if case["ham"] == "ising" else (0, 1 << i, 0.25)
        xm.append(x)
        zm.append(z)
        cf.append(c)
    return np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64), np.array(cf)


def _measured(case, seed):
    """The marginal's qubits and the samples' uniforms."""
    rng = np.random.default_rng(seed + 1)
    return [int(q) for q in rng.permutation(case["n"])[:case["m"]]], rng.random(case["shots"])


def _batch(case, seed):
    rng = np.random.default_rng(seed)
    nq = rng.integers(case["nlo"], case["nhi"] + 1, size=case["count"])
    return nq, [rng.uniform(0, 2 * np.pi, size=(LAYERS, int(n), 2)) for n in nq]


def _state(case, n, seed):
    st = qe.State(n, case["dtype"])
    if case["dtype"] == "c128" and case["arith"] == "df64":
        st.set_arith(qe.ARITH_DF64)
    if case.get("max_k"):
        st.set_policy(qe.POLICY_AUTO, case["max_k"])
    st.tensor.copy_(_amplitudes(n, seed, _real(case)))
    return st


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        nq, angles = _batch(case, seed)
        b = qe.Batch(nq, angles, HX, case["dtype"])
        if case["dtype"] == "c128" and case["arith"] == "fp64":
            b.set_arith(qe.ARITH_FP64)
        return {"kind": kind, "batch": b}
    n = case["nsys"] + case["b"] if kind == "qpe" else case["n"]
    s = {"kind": kind, "case": case, "st": _state(case, n, seed)}
    if kind == "circuit":
        s["gates"] = [(np.array(q, dtype=np.int32), np.ascontiguousarray(U)) for q, U in _circuit(n, case["depth"], seed)]
    elif kind == "add":
        s["qubits"], s["c"] = _register(case), _constant(case, seed)
    elif kind == "muldiv":
        s["regs"] = _registers(case)
    elif kind == "observe":
        s["ham"] = _hamiltonian(case)
        s["qubits"], s["u"] = _measured(case, seed)
    elif kind == "qpe":
        u = qe.State(2 * case["nsys"], "c128")
        u.init_identity(case["nsys"])
        for q, U in _trotter(case["nsys"], seed):
            u.apply_gate(q, U)
        u.flush()
        s["u"] = u
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        return s["batch"].run()
    st, case = s["st"], s["case"]
    if kind == "circuit":
        for q, U in s["gates"]:
            st.apply_gate(q, U)
        st.flush()
    elif kind == "qft":
        st.apply_qft(case["lo"], case["m"], case["inverse"])
    elif kind == "add":
        st.add_const(s["qubits"], s["c"])
    elif kind == "muldiv":
        st.mul(*s["regs"])
        st.div(*s["regs"])
    elif kind == "qpe":
        st.qpe_emulate(case["nsys"], case["b"], s["u"])
    else:
        return {"energy": np.array([st.expectation(*s["ham"])]), "probs": st.probs(s["qubits"]), "shots": st.sample(s["u"])}
    return st.tensor


def work(case):
    kind = case["kind"]
    amp = 16 if case["dtype"] == "c128" else 8
    if kind == "batch":
        # the mean circuit of the range: matrices in, energy out; a rotation
        # of each qubit costs 6 flops an amplitude and layer, a phase 6 a layer
        sizes = range(case["nlo"], case["nhi"] + 1)
        mean = sum(LAYERS * 2.0 ** n * (6 * n + 6) + 2.0 ** n * (4 + 4 * n) for n in sizes) / len(sizes)
        angles = sum(LAYERS * n * 16.0 for n in sizes) / len(sizes)
        return {"bytes": case["count"] * (angles + 8), "flops": case["count"] * mean}
    if kind == "qpe":
        D, b = 2.0 ** case["nsys"], case["b"]
        # squarings, controlled products on half the rows each, the Fourier transform
        flops = 8 * D ** 3 * (b - 1) + b * 8 * D * D * 2.0 ** (b - 1) + 5 * b * D * 2.0 ** b
        return {"bytes": amp * (D * D + 2 * D * 2.0 ** b), "flops": flops}
    N = 2.0 ** case["n"]
    if kind == "circuit":
        # 14 flops an amplitude for each dense one-qubit gate; CNOTs only move
        return {"bytes": 2 * amp * N, "flops": case["depth"] * case["n"] * 14 * N}
    if kind == "qft":
        return {"bytes": 2 * amp * N, "flops": 5 * case["m"] * N}
    if kind == "add":
        return {"bytes": 2 * amp * N, "flops": 0}
    if kind == "muldiv":
        return {"bytes": 2 * 2 * amp * N, "flops": 0}
    # every amplitude's weight, and two products a pair for each term that flips bits
    flips = case["n"] if case["ham"] == "ising" else 2 * (case["n"] - 1)
    return {"bytes": amp * N, "flops": N * (6 + 2 * flips)}


# ---------------------------------------------------------------- exact
def _vector(case, n, seed):
    x = _amplitudes(n, seed, _real(case)).double()
    return torch.view_as_complex(x.view(-1, 2))


def _flat(psi):
    return torch.view_as_real(psi.reshape(-1)).reshape(-1)


def _apply1(psi, q, U):
    """U on qubit q of the last axis' index, in place."""
    v = psi.view(-1, 2, 1 << q)
    a, b = v[:, 0].clone(), v[:, 1].clone()
    v[:, 0] = complex(U[0, 0]) * a + complex(U[0, 1]) * b
    v[:, 1] = complex(U[1, 0]) * a + complex(U[1, 1]) * b


def _cnot(psi, target, control):
    hi, lo = max(target, control), min(target, control)
    v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
    a, b = (v[:, 1, :, 0], v[:, 1, :, 1]) if control == hi else (v[:, 0, :, 1], v[:, 1, :, 1])
    t = a.clone()
    a.copy_(b)
    b.copy_(t)


def _apply(psi, gates):
    for q, U in gates:
        if len(q) == 1:
            _apply1(psi, q[0], U)
        else:
            _cnot(psi, q[0], q[1])


def _fourier(psi, lo, m, inverse):
    v = psi.view(-1, 1 << m, 1 << lo)
    if lo == 0:
        v = v.squeeze(-1)
        return (torch.fft.fft if inverse else torch.fft.ifft)(v, dim=1, norm="ortho").reshape(-1)
    out = torch.empty_like(v)
    for h in range(0, v.shape[0], max(1, (1 << 24) >> (m + lo))):
        part = slice(h, h + max(1, (1 << 24) >> (m + lo)))
        t = v[part].transpose(1, 2).contiguous()
        out[part] = (torch.fft.fft if inverse else torch.fft.ifft)(t, dim=2, norm="ortho").transpose(1, 2)
    return out.reshape(-1)


def _value(x, qubits):
    r = torch.zeros_like(x)
    for j, q in enumerate(qubits):
        r |= ((x >> q) & 1) << j
    return r


def _with_value(x, qubits, r):
    mask = sum(1 << q for q in qubits)
    x = x & ~mask
    for j, q in enumerate(qubits):
        x |= ((r >> j) & 1) << q
    return x


def _moved(psi, place):
    """The amplitude at x goes to place(x), a part of the indices at a time."""
    out = torch.empty_like(psi)
    step = 1 << 26
    for b in range(0, psi.numel(), step):
        x = torch.arange(b, min(b + step, psi.numel()), device=psi.device)
        out[place(x)] = psi[b:b + step]
    return out


def _divided(x, qa, qb, qc):
    N = len(qa)
    a, b, c = _value(x, qa), _value(x, qb), _value(x, qc)
    for i in range(N - 1, -1, -1):
        c = c ^ (((b != 0) & (a >= (b << i))).long() << i)
        a = torch.where(((c >> i) & 1) == 1, (a - (b << i)) & ((1 << N) - 1), a)
    return _with_value(_with_value(x, qa, a), qc, c)


def _dot(a, b):
    """Re sum conj(a) b, in parts."""
    a, b = torch.view_as_real(a.contiguous()).reshape(-1), torch.view_as_real(b.contiguous()).reshape(-1)
    return float(torch.stack([(x * y).sum() for x, y in zip(a.split(1 << 26), b.split(1 << 26))]).sum())


def _energy(psi, case):
    n, e = case["n"], 0.0
    p = psi.real.square() + psi.imag.square()
    for xm, zm, cf in zip(*(v.tolist() for v in _hamiltonian(case))):
        bits = [q for q in range(n) if ((xm | zm) >> q) & 1]
        lo = bits[0]
        if not xm:
            v = p.view(-1, 2 ** len(bits), 1 << lo).sum(dim=(0, 2)).tolist()
            e += cf * sum(w * (-1) ** bin(r).count("1") for r, w in enumerate(v))
        elif len(bits) == 1:
            v = psi.view(-1, 2, 1 << lo)
            e += cf * 2 * _dot(v[:, 0], v[:, 1])
        else:                     # XX or YY on neighbours
            v = psi.view(-1, 4, 1 << lo)
            e += cf * 2 * (_dot(v[:, 1], v[:, 2]) + (-1 if zm else 1) * _dot(v[:, 0], v[:, 3]))
    return e


def _ansatz_energies(case, seed):
    nq, angles = _batch(case, seed)
    out = np.zeros(case["count"])
    for n in sorted(set(int(v) for v in nq)):
        every = [c for c in range(case["count"]) if nq[c] == n]
        most = max(1, (1 << 26) >> n)
        for k in range(0, len(every), most):
            part = every[k:k + most]
            th = torch.tensor(np.stack([angles[c] for c in part]), device="cuda")
            psi = torch.zeros(len(part), 1 << n, dtype=torch.complex128, device="cuda")
            psi[:, 0] = 1
            x = torch.arange(1 << n, device="cuda")
            pairs = x & (x >> 1)
            odd = torch.zeros_like(x)
            for q in range(n):
                odd ^= (pairs >> q) & 1
            sign = (1 - 2 * odd).double()
            for l in range(LAYERS):
                for q in range(n):
                    t, f = th[:, l, q, 0].view(-1, 1, 1), th[:, l, q, 1].view(-1, 1, 1)
                    v = psi.view(len(part), -1, 2, 1 << q)
                    a, b = v[:, :, 0], v[:, :, 1]
                    c, s, ph = torch.cos(t / 2), torch.sin(t / 2), torch.polar(torch.ones_like(f), f / 2)
                    psi = torch.stack([(c * a - s * b) * ph.conj(), (s * a + c * b) * ph], dim=2).reshape(len(part), -1)
                psi = psi * sign
            p = psi.real.square() + psi.imag.square()
            e = torch.zeros(len(part), dtype=torch.float64, device="cuda")
            for q in range(n):
                v = torch.view_as_real(psi).view(len(part), -1, 2, 2 << q)
                e += 2 * HX * (v[:, :, 0] * v[:, :, 1]).sum(dim=(1, 2))
                if q + 1 < n:
                    w = p.view(len(part), -1, 4, 1 << q).sum(dim=(1, 3))
                    e += w[:, 0] - w[:, 1] - w[:, 2] + w[:, 3]
            out[part] = e.cpu().numpy()
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _ansatz_energies(case, seed)
    n = case["nsys"] + case["b"] if kind == "qpe" else case["n"]
    psi = _vector(case, n, seed)
    if kind == "circuit":
        _apply(psi, _circuit(n, case["depth"], seed))
    elif kind == "qft":
        psi = _fourier(psi, case["lo"], case["m"], case["inverse"])
    elif kind == "add":
        qubits, c = _register(case), _constant(case, seed)
        psi = _moved(psi, lambda x: _with_value(x, qubits, (_value(x, qubits) + c) & ((1 << len(qubits)) - 1)))
    elif kind == "muldiv":
        qa, qb, qc = _registers(case)
        most = (1 << case["N"]) - 1
        psi = _moved(psi, lambda x: _with_value(x, qc, (_value(x, qc) + _value(x, qa) * _value(x, qb)) & most))
        psi = _moved(psi, lambda x: _divided(x, qa, qb, qc))
    elif kind == "qpe":
        nsys, b = case["nsys"], case["b"]
        U = torch.eye(1 << nsys, dtype=torch.complex128, device="cuda")   # row j: column j of the matrix
        _apply(U.view(-1), _trotter(nsys, seed))
        for j in range(b):
            _apply1(psi, nsys + j, np.array([[1, 1], [1, -1]]) / math.sqrt(2.0))
        for j in range(b):
            v = psi.view(-1, 2, 1 << j, 1 << nsys)
            v[:, 1] = v[:, 1] @ U
            U = U @ U
        psi = _fourier(psi, nsys, b, True)
    else:
        qubits, _ = _measured(case, seed)
        p = psi.real.square() + psi.imag.square()
        for q in range(n - 1, -1, -1):       # the others summed out, from the top
            if q not in qubits:
                p = p.view(-1, 2, 1 << q).sum(dim=1)
        probs, kept = p.cpu().numpy(), sorted(qubits)
        where = [sum(((r >> j) & 1) << kept.index(q) for j, q in enumerate(qubits)) for r in range(probs.size)]
        return {"energy": np.array([_energy(psi, case)]), "probs": probs[where], "shots": None}
    return _flat(psi)
