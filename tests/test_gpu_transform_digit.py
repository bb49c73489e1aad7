"""One digit of a Fourier transform by itself, down to one tile a matrix, where
the blocks of a team outnumber the tiles of its matrix: every matrix is applied
to its own amplitudes.  Against the digit's definition in numpy; 56-bit rounding of
32 values and of 32 matrix entries leaves 64 2^-55 of the largest amplitude a
component."""
import ctypes as C

import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _reversed(v, bits):
    return sum(((v >> j) & 1) << (bits - 1 - j) for j in range(bits))


@pytest.mark.parametrize("n,q0,d,P", [(20, 0, 5, 8), (20, 3, 4, 8), (22, 2, 5, 10), (21, 0, 5, 8), (20, 1, 3, 5), (20, 0, 3, 8), (20, 12, 1, 0),
                                      (20, 18, 2, 0), (16, 4, 5, 0)])
def test_every_matrix_is_applied(n, q0, d, P):
    import torch
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(n, n + P)
    k = np.arange(1 << (P + d))
    roots = torch.tensor(np.exp(2j * np.pi * k / (1 << (P + d)))).cuda()
    with qe.State(n) as st:
        st.set(psi)
        digit = qe.load()["_ZN2qe21launch_dft_digit_c128EP8qe_stateiiiibPK7double2"]
        digit.argtypes, digit.restype = [C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_int, C.c_bool, C.c_void_p], None
        digit(st._h, 0, q0, d, P, True, roots.data_ptr())
        got = st.get()
        torch.cuda.synchronize()
    v = np.moveaxis(psi.reshape(-1, 1 << P, 1 << d, 1 << q0), 1, 0)
    ref = np.empty_like(v)
    rev = [_reversed(l, d) for l in range(1 << d)]
    for m in range(1 << P):
        prior = _reversed(m, P)
        U = np.array([[np.exp(2j * np.pi * ((kk * (prior + (l << P))) % (1 << (P + d))) / (1 << (P + d))) for kk in range(1 << d)]
                      for l in range(1 << d)]) * 2.0 ** (-0.5 * d)
        ref[m][:, rev] = np.einsum("lk,hkw->hlw", U, v[m])
    ref = np.moveaxis(ref, 0, 1).reshape(-1)
    bound = 64 * 2.0 ** -55 * float(np.max(np.abs(psi)))
    assert np.max(np.abs(got.view(float) - ref.view(float))) <= bound
