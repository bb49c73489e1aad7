"""The bit reversal of registers whose slices fit a tile, next to it and above it:
the simulated transform (which ends with the reversal) against the emulated one's
definition, every position of small registers, and states smaller than a tile."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

REGS = ([(n, lo, m) for n in (3, 7, 11, 13) for m in (2, 3, 6, 7) if m <= n for lo in sorted({0, 1, 2, (n - m) // 2, n - m}) if lo + m <= n] +
        [(14, lo, m) for lo in (0, 1, 3, 5) for m in (8, 9) ] + [(13, 0, 11), (13, 0, 12), (13, 1, 11), (14, 0, 13), (13, 4, 8)])


@pytest.mark.parametrize("n,lo,m", REGS)
@pytest.mark.parametrize("dtype,tol", [("c128", 1e-14), ("c64", 1e-5)])
def test_reversal(n, lo, m, dtype, tol):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n + m)
    v = psi.reshape(-1, 1 << m, 1 << lo)
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_SIMULATE)
        for inverse in (False, True):
            st.set(psi)
            st.apply_qft(lo, m, inverse)
            ref = (np.fft.fft if inverse else np.fft.ifft)(v, axis=1, norm="ortho").reshape(-1)
            assert np.max(np.abs(st.get() - ref)) < tol * m * 2.0 ** (-n / 2)
