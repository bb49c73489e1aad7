"""The digits of a Fourier transform and their groups (no GPU): over every
register of every state, the digits make up the register, a digit's matrix
serves at least 16 tiles of 2^12 amplitudes unless it is the first of its group,
and its roots fit a table of 2^20."""
import ctypes as C

import pytest

from paper_1604_06460_gb300 import build as B
from paper_1604_06460_gb300 import qe


@pytest.fixture(scope="module")
def digits():
    B.build()
    f = qe.load()["_ZN2qe10qft_digitsEiiPiS0_"]

    def plan(n, m):
        d, g = (C.c_int * 7)(), (C.c_int * 7)()
        k = f(n, m, d, g)
        return list(d[:k]), list(g[:k])
    return plan


@pytest.mark.parametrize("n", range(12, 35))
def test_groups_keep_their_limits(digits, n):
    for m in range(3, n + 1):
        d, g = digits(n, m)
        assert sum(d) == m and len(d) == -(-m // 5) and max(d) <= 5
        assert g[0] == 0 and all(0 <= b - a <= 1 for a, b in zip(g, g[1:]))
        for j in range(len(d)):
            P = sum(d[i] for i in range(j) if g[i] == g[j])
            assert P == 0 or (P <= n - 16 and P + d[j] <= 20), (n, m, d, g)
