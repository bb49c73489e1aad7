"""The host path of a gate: every accepted spelling of its arguments gives the
same state, what was refused stays refused, gates applied one by one (handed
over in lots while more are queued) keep their order, and threads marshal their
arguments independently."""
import threading

import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_argument_forms_agree():
    from paper_1604_06460_gb300 import qe
    U1, U2 = I.mat_h(), I.mat_cr(0.3) @ np.kron(I.mat_ry(0.2), I.mat_ry(0.9))
    psi = I.random_state(6, 1)
    ref = oracle.apply_gate(oracle.apply_gate(psi.copy(), (3,), U1), (4, 1), U2)
    forms = [((3,), U1, (4, 1), U2), ([3], U1.tolist(), [4, 1], U2.tolist()), (3, U1, np.array([4, 1]), U2),
             (np.int64(3), np.asfortranarray(U1), np.array([[4, 1]]), np.asfortranarray(U2)),
             (np.array([3], dtype=np.uint8), U1.real.copy(), (np.int32(4), 1), U2[::1, ::1])]
    for q1, A, q2, B in forms:
        with qe.State(6) as st:
            st.set(psi)
            st.apply_gate(q1, A)
            st.apply_gate(q2, B)
            assert np.max(np.abs(st.get() - ref)) < 1e-15


def test_refusals_stay():
    from paper_1604_06460_gb300 import qe
    with qe.State(6) as st:
        st.init_random(1)
        before = st.get()
        for q, U in [((0, 0), np.eye(4)), ((6,), np.eye(2)), ((-1,), np.eye(2)), ((0,), np.full((2, 2), np.nan)), ((), np.eye(1)),
                     (tuple(range(6)), np.eye(64))]:
            with pytest.raises(qe.QEError):
                st.apply_gate(q, np.asarray(U, dtype=np.complex128))
        with pytest.raises(ValueError):
            st.apply_gate((0,), np.eye(4, dtype=np.complex128))
        assert np.array_equal(st.get(), before)


@pytest.mark.parametrize("count", [1, 15, 16, 17, 40])
def test_gates_one_by_one_keep_their_order(count):
    from paper_1604_06460_gb300 import qe
    n = 7
    gates = I.random_circuit(n, 4, 5)[:count]
    psi = I.random_state(n, 2)
    ref = psi.copy()
    for g in gates:
        ref = oracle.apply_gate(ref, g.qubits, g.matrix)
    with qe.State(n) as st:
        st.set_policy(qe.POLICY_AUTO, 1)
        st.set(psi)
        for g in gates:
            st.apply_gate(g.qubits, g.matrix)
        assert np.max(np.abs(st.get() - ref)) < 1e-14
        assert st.stats()["gates_applied"] == count


def test_threads_marshal_independently():
    import torch
    from paper_1604_06460_gb300 import qe
    n, out = 8, {}

    def work(seed):
        torch.cuda.set_device(0)
        psi, gates = I.random_state(n, seed), I.random_circuit(n, 6, seed)
        with qe.State(n, stream=torch.cuda.Stream()) as st:
            st.set(psi)
            for g in gates:
                st.apply_gate(g.qubits, g.matrix)
            out[seed] = st.get()

    ts = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    for seed in range(4):
        ref = I.random_state(n, seed)
        for g in I.random_circuit(n, 6, seed):
            ref = oracle.apply_gate(ref, g.qubits, g.matrix)
        assert np.max(np.abs(out[seed] - ref)) < 1e-14
