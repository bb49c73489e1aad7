"""Emulated multiplication and division where their path changes: planes of one
tile and just above it, register widths around them, registers with free qubits
below them, interleaved and unordered registers, and states smaller than a
tile.  Bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def contiguous(N, lo):
    return [list(range(lo + k * N, lo + (k + 1) * N)) for k in (2, 1, 0)]


def interleaved(N, n, seed):
    p = [int(v) for v in np.random.default_rng(seed).permutation(n)[:3 * N]]
    return p[:N], p[N:2 * N], p[2 * N:]


REGS = ([(n, contiguous(N, lo)) for n, N, lo in
         [(3, 1, 0), (6, 2, 0), (12, 4, 0), (18, 6, 0), (19, 6, 1), (21, 7, 0), (22, 7, 1), (20, 6, 2), (20, 5, 5), (16, 2, 9)]] +
        [(n, interleaved(N, n, N)) for n, N in [(11, 3), (18, 6), (21, 7), (20, 4)]] +
        [(21, (list(range(7)), list(range(7, 14)), list(range(14, 21))))])


@pytest.mark.parametrize("n,regs", REGS, ids=lambda v: str(v) if isinstance(v, int) else "")
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_mul_div_paths(n, regs, dtype):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.set(psi)
        st.mul(*regs)
        assert np.array_equal(st.get().astype(np.complex128), oracle.mul(psi.copy(), *regs))
        st.set(psi)
        st.div(*regs)
        assert np.array_equal(st.get().astype(np.complex128), oracle.div(psi.copy(), *regs))
