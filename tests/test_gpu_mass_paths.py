"""Marginals and samples around the sizes where their kernels split: registers
on both sides of qubit 8, states smaller than one block row, components of very
different size, sparse states.  Sums of n non-negative terms, each exact to
2^-50 of its group's largest, in FP64: 1e-13 of the total is above any rounding
of 2^20 such terms in groups; bins of zero probability stay exactly zero."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SETS = [(1, [0]), (3, [2, 0]), (7, [6, 1]), (8, list(range(8))), (9, [8]), (9, [8, 3, 0]), (10, [9, 8, 1]), (12, [4, 11]),
        (13, [12, 5, 8, 0, 10]), (16, list(range(15, -1, -1))), (17, [7, 8]), (20, [19, 3, 8, 15]), (20, list(range(4, 16)))]


@pytest.mark.parametrize("arith", ["fp64", "df64"])
@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,qubits", SETS)
def test_probs_paths(n, qubits, dtype, arith):
    from paper_1604_06460_gb300 import qe
    rng = np.random.default_rng(n)
    psi = I.random_state(n, n) * 2.0 ** rng.integers(-30, 1, 1 << n)
    psi[rng.random(1 << n) < 0.25] = 0
    psi /= np.linalg.norm(psi)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    with qe.State(n, dtype) as st:
        st.set_arith(getattr(qe, "ARITH_" + arith.upper()))
        st.set(psi)
        p, nrm = st.probs(qubits), st.norm2()
    ref = oracle.probs(psi, qubits)
    assert np.all((p == 0) == (ref == 0))
    assert np.max(np.abs(p - ref)) < 1e-13
    assert abs(nrm - ref.sum()) < 1e-13


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("n,every", [(17, 1), (18, 4099), (18, 512), (20, 70001), (16, 37)])
def test_sparse_samples(n, every, dtype):
    from paper_1604_06460_gb300 import qe
    psi = np.zeros(1 << n, dtype=np.complex128)
    at = np.arange(every // 2, 1 << n, every)
    psi[at] = np.random.default_rng(n).standard_normal(at.size) + 0.1j
    psi /= np.linalg.norm(psi)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    u = np.concatenate([[0.0, 1 - 2.0 ** -53], np.random.default_rng(3).random(3000)])
    with qe.State(n, dtype) as st:
        st.set(psi)
        got = np.asarray(st.sample(u))
    p = np.abs(psi[got]) ** 2
    assert np.all(p > 0)
    top = np.cumsum(np.abs(psi) ** 2)
    total = top[-1]
    # the sample's interval of the distribution holds the target, to rounding
    assert np.all(top[got] >= u * total - 1e-13)
    assert np.all(top[got] - p <= u * total + 1e-13)
