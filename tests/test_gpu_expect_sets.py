"""Expectations of large states by register sets: terms of one to four X/Y
qubits anywhere, Z parts everywhere, Z-only masks of every kind, several
weights, more terms than a launch holds; against the oracle, 1e-13 of
sum |c| ||psi||^2 as the other fixed-point kernel (products exact to 2^-51 of the
largest in 512 amplitudes; sums of 2^20 such in FP64)."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _register_sets(monkeypatch):
    monkeypatch.setenv("QE_EXPECT_TILE", "3")      # whichever path is cheaper


def _energy(n, psi, xm, zm, cf, dtype, arith):
    from paper_1604_06460_gb300 import qe
    with qe.State(n, dtype) as st:
        st.set_arith(getattr(qe, "ARITH_" + arith.upper()))
        st.set(psi)
        st.profile(True)
        e = st.expectation(np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64), np.array(cf, dtype=float))
        prof = st.profile_read()
    assert ("expect_fx" if dtype == "c128" else "expect_rounds") in prof and "expect_tile" not in prof, prof
    return e


def _chain(n):
    xm, zm, cf = [], [], []
    for i in range(n - 1):
        p = 3 << i
        xm += [p, p, 0]; zm += [0, p, p]; cf += [1.0, 0.9, 1.1]
    for i in range(n):
        xm += [0, 1 << i]; zm += [1 << i, 0]; cf += [0.25, 0.7]
    return xm, zm, cf


def _fields(n):
    # single X on two, three and four qubits of a set, of several weights and signs, some twice
    xm, zm, cf = [], [], []
    for i in range(n):
        for w in ([0.7], [0.7, -0.4], [-0.4], [0.7, 0.7, 1.3])[(i * 7 // 4) % 4]:
            xm.append(1 << i); zm.append(0); cf.append(w)
    return xm, zm, cf


def _mixed(n, seed, count=90):
    rng = np.random.default_rng(seed)
    xm, zm, cf = [], [], []
    weights = [0.5, -1.25, 0.5, 2.0]
    for pat in range(1, 16):                       # every pattern of qubits 0 to 3 and of four others
        for sh in (0, 5, n - 4):
            xm.append(pat << sh); zm.append(int(rng.integers(0, 1 << n))); cf.append(weights[pat % 4])
    for _ in range(6):
        qs = rng.choice(n, size=int(rng.integers(1, 5)), replace=False)
        xm.append(int(sum(1 << int(q) for q in qs))); zm.append(int(rng.integers(0, 1 << n))); cf.append(-0.75)
    for _ in range(count):
        xm.append(0); zm.append(int(rng.integers(0, 1 << n))); cf.append(weights[int(rng.integers(0, 4))])
    for i in range(n - 3):
        xm.append(0); zm.append((1 << i) | (1 << (i + 3))); cf.append(0.3)
    return xm, zm, cf


CASES = [(17, "chain"), (18, "fields"), (19, "fields"), (18, "mixed"), (20, "chain"), (21, "mixed"), (20, "mixed"), (22, "chain")]


@pytest.mark.parametrize("dtype,arith", [("c128", "fp64"), ("c128", "df64"), ("c64", "fp64")])
@pytest.mark.parametrize("n,kind", CASES)
def test_expectation_register_sets(n, kind, dtype, arith):
    xm, zm, cf = _chain(n) if kind == "chain" else _fields(n) if kind == "fields" else _mixed(n, n)
    rng = np.random.default_rng(n)
    psi = I.random_state(n, n)
    psi = (psi.reshape(-1, 128) * 2.0 ** rng.integers(-40 if dtype == "c128" else -20, 1, (1 << n) // 128)[:, None]).reshape(-1)
    psi[: 1 << 12] = 0
    psi /= np.linalg.norm(psi)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    e = _energy(n, psi, xm, zm, cf, dtype, arith)
    ref = oracle.expectation(psi, np.array(xm, dtype=np.uint64), np.array(zm, dtype=np.uint64), np.array(cf))
    assert abs(e - ref) <= 1e-13 * float(np.sum(np.abs(cf))), (e, ref)


def test_expectation_register_sets_not_a_number():
    n = 20
    psi = I.random_state(n, 1)
    psi[12345] = np.nan
    xm, zm, cf = _chain(n)
    assert np.isnan(_energy(n, psi, xm, zm, cf, "c128", "fp64"))
