"""Circuits of a warp each (up to eight qubits: one to eight amplitudes a lane)
alone and among larger ones, one to nine layers, angles where a rotation's
outputs trade places; against the oracle, tolerances those of the batch's other
tests."""
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


@pytest.mark.parametrize("layers", [1, 2, 9])
@pytest.mark.parametrize("ns", [[1], [7], [8], [1, 2, 3, 4, 5, 6, 7], [7, 8, 5, 13, 6, 3, 7, 7, 2, 8], [6, 1, 12, 8, 5],
                                [7] * 310])
@pytest.mark.parametrize("dtype,arith,tol", [("c128", 0, 2.0 ** -46), ("c128", 1, 1e-11), ("c64", None, 2e-4)])
def test_tiny_circuits(ns, layers, dtype, arith, tol):
    from paper_1604_06460_gb300 import qe
    rng = np.random.default_rng(sum(ns) + layers)
    angles = [rng.uniform(-2 * np.pi, 2 * np.pi, size=(layers, n, 2)) for n in ns]
    angles[-1][:, :, 0] = rng.choice([0.0, np.pi / 2, np.pi, -np.pi / 2, 3 * np.pi], size=angles[-1].shape[:2])
    with qe.Batch(ns, angles, 0.7, dtype) as b:
        if arith is not None:
            b.set_arith(arith)
        e = b.run()
        assert np.array_equal(e, b.run())
    some = sorted({*range(min(len(ns), 10)), len(ns) - 1})
    ref = np.array([_energy(ns[i], angles[i], 0.7) for i in some])
    assert np.max(np.abs(e[some] - ref)) < tol
