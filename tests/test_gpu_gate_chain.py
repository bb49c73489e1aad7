"""Elementwise gates one after another on a stream: each kernel starts before
the one before has ended and waits for it, whatever the sizes of the two (one
block, fewer blocks than SMs, several waves) and whatever kind follows.  The
chain's result equals the same gates with a synchronisation after each, bit
for bit."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,arith", [("c128", "fp64"), ("c128", "df64"), ("c64", "fp64")])
@pytest.mark.parametrize("n", [3, 9, 13, 18, 21])
def test_chained_gates_bit_identical(n, dtype, arith):
    from paper_1604_06460_gb300 import qe
    rng = np.random.default_rng(n)
    cnot = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], dtype=complex)
    gates = []
    for _ in range(120):
        k = int(rng.integers(0, 4))
        q = [int(v) for v in rng.permutation(n)]
        u, _ = np.linalg.qr(rng.standard_normal((4, 4)) + 1j * rng.standard_normal((4, 4)))
        v, _ = np.linalg.qr(rng.standard_normal((2, 2)) + 1j * rng.standard_normal((2, 2)))
        gates.append([(q[:1], v), (q[:2], u), (q[:2], cnot), (q[:1], np.diag(np.exp(1j * rng.random(2))))][k])
    psi = I.random_state(n, n)
    out = []
    for wait in (False, True):
        with qe.State(n, dtype) as st:
            st.set_arith(getattr(qe, "ARITH_" + arith.upper()))
            st.set_policy(qe.POLICY_AUTO, max_k=1)
            st.set(psi.astype(np.complex64) if dtype == "c64" else psi)
            for q, m in gates:
                st.apply_gate(q, m)
                if wait:
                    st.flush()
                    st.sync()
            out.append(st.get())
    assert np.array_equal(out[0], out[1])
