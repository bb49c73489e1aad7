"""Phase estimation where its products change path: system registers around the
smallest that runs on the tensor cores, few and many controlled rows, and
repeated calls on states of different sizes (kept workspaces)."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def reference(psi, U, nsys, b, n):
    v = psi.reshape([2] * (n - nsys) + [1 << nsys])   # axis 0: the top ancilla or spectator
    for j in range(b):
        a = n - nsys - 1 - j
        v = np.moveaxis(v, a, 0)
        v = np.stack([v[0] + v[1], v[0] - v[1]]) / np.sqrt(2.0)
        v = np.moveaxis(v, 0, a)
    P = U.copy()
    for j in range(b):
        a = n - nsys - 1 - j
        v = np.moveaxis(v, a, 0).copy()
        v[1] = v[1] @ P.T
        v = np.moveaxis(v, 0, a)
        P = P @ P
    v = np.ascontiguousarray(v).reshape(-1, 1 << b, 1 << nsys)
    return np.fft.fft(v, axis=1, norm="ortho").reshape(-1)


@pytest.mark.parametrize("nsys,b,extra", [(5, 3, 0), (6, 1, 0), (6, 3, 1), (6, 8, 0), (7, 2, 0), (7, 5, 2), (8, 4, 0), (8, 8, 0)])
def test_qpe_paths(nsys, b, extra):
    from paper_1604_06460_gb300 import qe
    n = nsys + b + extra
    psi = I.random_state(n, n)
    U = np.eye(1 << nsys, dtype=np.complex128)
    gates = I.tfim_trotter_step(nsys, 0.3)
    with qe.State(2 * nsys) as u, qe.State(n) as st:
        u.init_identity(nsys)
        for g in gates:
            u.apply_gate(g.qubits, g.matrix)
        u.flush()
        U = u.get().reshape(1 << nsys, 1 << nsys).T.copy()
        for _ in range(2):
            st.set(psi)
            st.qpe_emulate(nsys, b, u)
            got = st.get()
            # b controlled products and squarings, each within a few units of
            # 2^-53 sqrt(2^nsys) of its norm, doubled in relative size by every squaring
            assert np.max(np.abs(got - reference(psi, U, nsys, b, n))) < 2.0 ** -53 * 4 * (1 << b) * 2 ** (nsys / 2)
