"""Transforms of states whose branches (assignments of the qubits outside the
register) differ in size by 2^30: each branch is transformed to rounding of
its own norm.  Tensor-core digits: an output is within 2^-50 of the product of its
row's and its matrix row's scales, at most four times the largest amplitude of
the row and 2^-5/2, hence 2^-47 of the branch's norm a digit.  Elementwise FP64
stays below that, elementwise double-float (47 bits) below 2^-42 a pass of
stages."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FP64 = ([(20, lo, m) for m in range(5, 19) for lo in sorted({0, (20 - m) // 2, 20 - m})] +
        [(19, 1, 17), (21, 0, 19), (22, 0, 13), (22, 5, 16), (23, 2, 11), (24, 1, 22)])
DF64 = [(22, 0, 5), (22, 9, 5), (22, 1, 4), (22, 0, 3), (22, 18, 4), (23, 0, 22), (23, 6, 17), (23, 3, 12), (23, 11, 12)]


@pytest.mark.parametrize("n,lo,m,arith", [(*r, 0) for r in FP64] + [(*r, 1) for r in DF64])
def test_branches_keep_their_own_precision(n, lo, m, arith):
    from paper_1604_06460_gb300 import qe
    rng = np.random.default_rng(n + m)
    psi = I.random_state(n, n + m).reshape(-1, 1 << m, 1 << lo)
    psi = psi * np.where(rng.random((psi.shape[0], 1, 1 << lo)) < 0.5, 1.0, 2.0 ** -30)
    ref = np.fft.ifft(psi, axis=1, norm="ortho")
    with qe.State(n) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.set_arith(arith)
        st.set(psi.reshape(-1))
        st.apply_qft(lo, m)
        got = st.get().reshape(psi.shape)
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.max(err) < -(-m // 5) * (2.0 ** -47 if arith == 0 else 2.0 ** -42)
