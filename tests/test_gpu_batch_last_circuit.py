"""A batch whose last circuit is larger than a tile: its final read-only pass
comes after the last layer, and the flip masks, one a layer, end the
allocation that holds them.  One to three layers, alone and after a small
circuit, each arithmetic, at tiles that leave one and several tile bits;
tolerances those of the batch's other tests."""
import numpy as np
import pytest

import oracle
from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _energy(n, angles, hx):
    psi = oracle.zero_state(n)
    for layer in angles:
        for q in range(n):
            oracle.apply_gate(psi, (q,), I.mat_ry(layer[q, 0]), inplace=True)
            oracle.apply_gate(psi, (q,), I.mat_rz(layer[q, 1]), inplace=True)
        for q in range(n - 1):
            g = I.cz(q, q + 1)
            oracle.apply_gate(psi, g.qubits, g.matrix, inplace=True)
    return oracle.expectation(psi, *I.tfim_terms(n, hx))


@pytest.mark.parametrize("layers", [1, 2, 3])
@pytest.mark.parametrize("ns", [[9], [4, 11], [14]])
@pytest.mark.parametrize("dtype,arith,tol", [("c128", 0, 2.0 ** -46), ("c128", 1, 1e-11), ("c64", None, 2e-4)])
def test_last_circuit_above_a_tile(ns, layers, dtype, arith, tol):
    from paper_1604_06460_gb300 import qe
    rng = np.random.default_rng(ns[-1] + layers)
    angles = [rng.uniform(0, 2 * np.pi, size=(layers, n, 2)) for n in ns]
    with qe.Batch(ns, angles, 0.7, dtype) as b:
        if ns[-1] < 14:
            b.set_plan(8, 1, 128)
        if arith is not None:
            b.set_arith(arith)
        e = b.run()
        assert np.array_equal(e, b.run())
    ref = np.array([_energy(n, a, 0.7) for n, a in zip(ns, angles)])
    assert np.max(np.abs(e - ref)) < tol
