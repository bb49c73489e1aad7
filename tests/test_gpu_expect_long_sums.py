"""Sums of many terms on large states, where the plan uses its tables: strings of
one to four X/Y qubits with Z parts, many times the same sets, masks of many and
of few weights, just below and above the length at which the tables begin.
Against the sum of its parts."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _terms(n, count, seed):
    rng = np.random.default_rng(seed)
    xm, zm = np.zeros(count, dtype=np.uint64), rng.integers(0, 1 << n, count).astype(np.uint64)
    for i in range(count):
        k = int(rng.integers(0, 5))
        xm[i] = sum(1 << int(q) for q in rng.choice(n if i % 3 else 9, size=k, replace=False))
    return xm, zm, np.where(rng.random(count) < 0.5, 0.5, rng.normal(size=count))


@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("path", [None, "3"])
@pytest.mark.parametrize("count", [250, 330, 2500])
def test_long_sums(count, path, dtype, monkeypatch):
    from paper_1604_06460_gb300 import qe
    if path:
        monkeypatch.setenv("QE_EXPECT_TILE", path)
    n = 17
    xm, zm, cf = _terms(n, count, count)
    with qe.State(n, dtype) as st:
        st.set(I.random_state(n, 8))
        e = st.expectation(xm, zm, cf)
        parts = sum(st.expectation(xm[i:i + 20], zm[i:i + 20], cf[i:i + 20]) for i in range(0, count, 20))
    assert abs(e - parts) <= 1e-13 * float(np.sum(np.abs(cf)))
