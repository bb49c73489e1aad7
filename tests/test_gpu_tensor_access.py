"""The tensor-core kernels' memory access where its form changes: blocks with
and without qubits 0 and 1 (pairs and quads of columns that are neighbours in
memory), qubits given in any order, narrower blocks widened by idle qubits, and
Fourier transforms whose digits are 3..5 qubits wide, meet matrices that depend
on the qubits above them, or are one digit alone."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def unitary(k, seed):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((1 << k, 1 << k)) + 1j * rng.standard_normal((1 << k, 1 << k))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))[None, :]


BLOCKS = [(0, 1, 2, 3, 4), (4, 2, 0, 3, 1), (0, 2, 4, 6, 8), (1, 0, 13, 5, 9), (13, 0, 7, 6, 5), (1, 2, 3, 4, 5),
          (9, 10, 11, 12, 13), (5, 6, 7, 8, 9), (0, 5, 12), (12, 1, 0), (6, 3, 9, 13), (0, 1, 2, 3), (13, 5, 6)]


@pytest.mark.parametrize("qubits", BLOCKS)
@pytest.mark.parametrize("dtype,arith,tol", [("c128", 0, 16 * 2.0 ** -53), ("c128", 1, 1e-12), ("c64", None, 2e-5)])
def test_block_access_forms(qubits, dtype, arith, tol):
    from paper_1604_06460_gb300 import qe
    n, U = 14, unitary(len(qubits), sum(qubits))
    psi = I.random_state(n, 11)
    ref = oracle.apply_gate(psi.copy(), qubits, U)
    with qe.State(n, dtype) as st:
        if arith is not None:
            st.set_arith(arith)
        st.set(psi)
        st.apply_gate(qubits, U)
        got = st.get()
    # FP64: a few units of a 32-amplitude group's norm (here up to 32 / 2^7)
    assert np.max(np.abs(got - ref)) < tol


REGISTERS = [(12, 0, 12), (12, 9, 3), (12, 0, 3), (13, 4, 7), (14, 0, 13), (20, 0, 5), (20, 15, 5), (20, 0, 4),
             (20, 9, 11), (20, 1, 17), (21, 0, 21), (21, 3, 14), (22, 5, 17)]


@pytest.mark.parametrize("n,lo,m", REGISTERS)
@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("dtype,arith,tol", [("c128", 0, 1e-14), ("c128", 1, 1e-12), ("c64", None, 1e-5)])
def test_qft_digits(n, lo, m, inverse, dtype, arith, tol):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, 7 * n + m)
    v = psi.reshape(-1, 1 << m, 1 << lo)
    ref = (np.fft.fft if inverse else np.fft.ifft)(v, axis=1, norm="ortho").reshape(-1)
    with qe.State(n, dtype) as st:
        if arith is not None:
            st.set_arith(arith)
        st.set_policy(qe.POLICY_EMULATE)
        st.set(psi)
        st.apply_qft(lo, m, inverse)
        got = st.get()
    # errors grow with the passes, not with n: relative to the state's rms
    rms = 2.0 ** (-n / 2)
    assert np.max(np.abs(got - ref)) < tol * rms * m
