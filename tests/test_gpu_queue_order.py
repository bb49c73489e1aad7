"""Queued gates touch the state at the next flush and not before, however many
they are and whatever the fusion width: the caller may read and write a borrowed
buffer between the two."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_k", [0, 1])
@pytest.mark.parametrize("count", [15, 16, 40])
def test_gates_wait_for_the_flush(count, max_k):
    import torch
    from paper_1604_06460_gb300 import qe
    n = 7
    gates = I.random_circuit(n, 4, 5)[:count]
    first, second = I.random_state(n, 2), I.random_state(n, 3)
    with qe.State(n) as st:
        st.set_policy(qe.POLICY_AUTO, max_k)
        st.set(first)
        for g in gates:
            st.apply_gate(g.qubits, g.matrix)
        torch.cuda.synchronize()
        assert np.array_equal(st.tensor.cpu().numpy().view(complex), first)
        st.tensor.copy_(torch.tensor(second.view(float)))
        got = st.get()
    for g in gates:
        second = oracle.apply_gate(second, g.qubits, g.matrix)
    assert np.max(np.abs(got - second)) < 1e-14
