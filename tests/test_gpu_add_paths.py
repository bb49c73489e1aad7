"""The emulated addition of a constant where its path changes: slices around the
cluster sizes, and registers at the bottom of the state too large for them
(rotation of small slices, then the upper bits with the carry).  Bit-exact."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [(18, 0, 15), (18, 0, 16), (18, 1, 16), (18, 0, 17), (18, 0, 18), (20, 0, 18), (20, 2, 18), (19, 4, 15),
         (21, 0, 20), (20, 3, 14), (17, 0, 17)]
SPLIT = [("c128", 24, 0, 18), ("c128", 24, 1, 20), ("c128", 24, 0, 24), ("c128", 24, 2, 18), ("c64", 25, 0, 19),
         ("c64", 25, 0, 17), ("c64", 25, 1, 18), ("c64", 25, 2, 20), ("c64", 25, 3, 18)]


@pytest.mark.parametrize("n,lo,m", CASES)
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_add_const_paths(n, lo, m, dtype):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    top = 1 << m
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_EMULATE)
        for c in (1, 2, 3, 4096, 4097, 8192, top // 2, top // 2 + 8, top - 1, top - 4096, 0x2A5F3 % top):
            st.set(psi)
            st.add_const(list(range(lo, lo + m)), c)
            ref = np.roll(psi.reshape(-1, top, 1 << lo), c % top, axis=1).reshape(-1)
            assert np.array_equal(st.get().astype(np.complex128), ref), c


@pytest.mark.parametrize("dtype,n,lo,m", SPLIT)
def test_add_const_split_registers(dtype, n, lo, m):
    from paper_1604_06460_gb300 import qe
    top = 1 << m
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.init_random(n)
        psi = st.get().reshape(-1, top, 1 << lo)
        at = 0
        for c in (1, 4096, 16384 >> lo, top // 2 + 3, top - 1, 0x2A5F3A7 % top):
            st.add_const(list(range(lo, lo + m)), c)
            at = (at + c) % top
            assert np.array_equal(st.get(), np.roll(psi, at, axis=1).reshape(-1)), c
