"""Transforms whose digits fall into several groups of unequal length; against
numpy, 1e-14 of the state's rms a register qubit as the other digit tests."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lo,m", [(19, 0, 11), (19, 8, 11), (20, 3, 14), (20, 0, 18), (24, 0, 23), (24, 1, 22), (25, 1, 24)])
def test_qft_groups(n, lo, m):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n + m)
    ref = np.fft.ifft(psi.reshape(-1, 1 << m, 1 << lo), axis=1, norm="ortho").reshape(-1)
    with qe.State(n) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.set(psi)
        st.apply_qft(lo, m)
        got = st.get()
    assert np.max(np.abs(got - ref)) < 1e-14 * 2.0 ** (-n / 2) * m
