"""Additions to slices of 1 and 2 MB where the device runs no clusters of sixteen
blocks (pretended): the portable clusters and the other paths take them, bit for
bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("without", [False, True])
@pytest.mark.parametrize("dtype,n,lo,m", [("c128", 18, 0, 16), ("c128", 17, 2, 14), ("c128", 18, 1, 16), ("c128", 24, 2, 15),
                                          ("c128", 25, 0, 17), ("c64", 19, 0, 17), ("c64", 18, 3, 15), ("c64", 25, 0, 18)])
def test_add_without_large_clusters(dtype, n, lo, m, without, monkeypatch):
    from paper_1604_06460_gb300 import qe
    if without:
        monkeypatch.setenv("QE_TEST_NO_CLUSTER16", "1")
    top = 1 << m
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.init_random(n)
        psi = st.get().reshape(-1, top, 1 << lo)
        at = 0
        for c in (1, 4096, top // 2, top - 1, 0x2A5F3A7 % top):
            st.add_const(list(range(lo, lo + m)), c)
            at = (at + c) % top
            assert np.array_equal(st.get(), np.roll(psi, at, axis=1).reshape(-1)), c
