"""An infinity or NaN among the inputs reaches the outputs that depend on it, and
only those: transforms on the tensor cores, where it makes its assignment of the
other qubits not finite, and phase estimation with few and many rows."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,lo,m,arith", [(20, 0, 7, 0), (20, 4, 11, 0), (21, 2, 17, 0), (20, 15, 5, 0), (22, 0, 5, 1), (23, 1, 19, 1)])
def test_transform(n, lo, m, arith, bad):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n + m)
    rng = np.random.default_rng(m)
    with qe.State(n) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.set_arith(arith)
        st.set(psi)
        st.apply_qft(lo, m)
        ref = st.get().reshape(-1, 1 << m, 1 << lo)
        h, k, l = (int(rng.integers(0, v)) for v in ref.shape)
        part = psi.reshape(ref.shape).view(float).reshape(*ref.shape, 2)
        part[h, k, l, m % 2] = bad
        st.set(psi)
        st.apply_qft(lo, m)
        got = st.get().reshape(ref.shape)
    finite = np.isfinite(got).any(axis=1)
    assert not finite[h, l]
    got[h, :, l] = ref[h, :, l]
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("nsys,b", [(6, 2), (7, 4), (6, 9)])
def test_phase_estimation(nsys, b):
    from paper_1604_06460_gb300 import qe
    n = nsys + b
    with qe.State(n) as st, qe.State(2 * nsys) as u:
        u.init_identity(nsys)
        psi = I.random_state(n, 5)
        psi[(1 << n) - 3] = np.nan       # the row of all ancillas set, before the Hadamards spread it
        st.set(psi)
        st.qpe_emulate(nsys, b, u)
        assert not np.isfinite(st.get()).any()
