"""The batch's rotations where their form changes: angles at which the two
outputs of a rotation trade places or not (multiples of pi/2 and next to
them), a single layer (the product state alone), one qubit, and tiles that
make one, two or more register groups a pass."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# edges of |tan(theta/2)| <= 1 and of the flips' parity
THETAS = [0.0, np.pi / 2, -np.pi / 2, np.pi, 3 * np.pi / 2, 2 * np.pi, np.pi / 2 + 1e-9, np.pi / 2 - 1e-9,
          np.pi + 1e-7, 5.0, -2.5, 1e-12]


def angles_of(n, layers, shift):
    a = np.empty((layers, n, 2))
    for l in range(layers):
        for q in range(n):
            a[l, q] = THETAS[(shift + 5 * l + 3 * q) % len(THETAS)], THETAS[(shift + 7 * l + q) % len(THETAS)]
    return a


def oracle_energy(n, angles, hx):
    psi = oracle.zero_state(n)
    for layer in angles:
        for q in range(n):
            oracle.apply_gate(psi, (q,), I.mat_ry(layer[q, 0]), inplace=True)
            oracle.apply_gate(psi, (q,), I.mat_rz(layer[q, 1]), inplace=True)
        for q in range(n - 1):
            g = I.cz(q, q + 1)
            oracle.apply_gate(psi, g.qubits, g.matrix, inplace=True)
    xm, zm, cf = I.tfim_terms(n, hx)
    return oracle.expectation(psi, xm, zm, cf)


@pytest.mark.parametrize("layers", [1, 2, 4])
@pytest.mark.parametrize("dtype,arith,tol", [("c128", 0, 2.0 ** -46), ("c128", 1, 1e-11), ("c64", None, 2e-4)])
@pytest.mark.parametrize("plan", [None, (7, 2, 128), (8, 1, 512)])
def test_batch_rotation_forms(layers, dtype, arith, tol, plan):
    from paper_1604_06460_gb300 import qe
    ns = [1, 2, 4, 6, 7, 8, 9, 10, 12, 13, 5]
    angles = [angles_of(n, layers, i) for i, n in enumerate(ns)]
    with qe.Batch(ns, angles, 0.7, dtype) as b:
        if plan is not None:
            b.set_plan(*plan)
        if arith is not None:
            b.set_arith(arith)
        e = b.run()
        assert np.array_equal(e, b.run())
    ref = np.array([oracle_energy(n, a, 0.7) for n, a in zip(ns, angles)])
    assert np.max(np.abs(e - ref)) < tol
