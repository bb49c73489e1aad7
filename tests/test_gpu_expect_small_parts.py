"""Terms that pair one large with one small amplitude (a nearly classical state),
where the products are native ones: complex128 terms across the triples of
qubits and all complex64 terms keep the relative digits of FP64 and of float
pairs (44 bits), whichever path takes them; also weights far apart, and a
complex64 state of small norm.  Against extended precision; a term's two large
products are rounded a few times, the sum of the others is below 2^-60 of them."""
import numpy as np
import pytest

from paper_1604_06460_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N = 18
TERMS = [[(12, 0, 1.0)], [(96, 0, 1.0), (96, 96, 0.9), (0, 96, 0.0)], [(0b1000010000100001, 0, -0.7)],
         [(1 << 17 | 4, 1 << 9, 1.3)], [(0b11000, 0b01000, 0.5)], [(3 << i, 0, 1.0) for i in range(N - 1)],
         [(12, 0, 1e-9), (96, 0, 1.0)]]


def _reference(psi, terms):
    e = np.longdouble(0)
    x = np.arange(psi.size)
    re, im = psi.real.astype(np.longdouble), psi.imag.astype(np.longdouble)
    for xm, zm, c in terms:
        p = x ^ xm
        sign = 1 - 2 * (np.bitwise_count(x & zm).astype(int) & 1)
        ny = bin(xm & zm).count("1") & 3
        # i^ny conj(a_p) a_x, real part
        v = re[p] * re + im[p] * im if ny % 2 == 0 else -(re[p] * im - im[p] * re)
        e += np.longdouble(c) * (v * sign).sum() * (-1 if ny >= 2 else 1)
    return e


@pytest.mark.parametrize("path", [None, "3"])
@pytest.mark.parametrize("terms", TERMS, ids=range(len(TERMS)))
@pytest.mark.parametrize("dtype,arith,scale,tol", [("c128", 0, 1.0, 1e-14), ("c64", 0, 1.0, 2.0 ** -40), ("c64", 0, 2.0 ** -24, 2.0 ** -40)])
def test_small_parts(dtype, arith, scale, tol, terms, path, monkeypatch):
    from paper_1604_06460_gb300 import qe
    if path:
        monkeypatch.setenv("QE_EXPECT_TILE", path)
    if dtype == "c128" and all(any(xm & ~(7 << t) == 0 for t in (0, 3, 6, 9)) for xm, _, _ in terms):
        pytest.skip("within the triples of qubits: fixed point")
    psi = I.random_state(N, 4) * 2.0 ** (N / 2) * 1e-10
    psi[0x1234] = 0.8 - 0.6j
    psi = psi * scale
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(complex)
    xm, zm, cf = (np.array(v, dtype=t) for v, t in zip(zip(*terms), (np.uint64, np.uint64, float)))
    with qe.State(N, dtype) as st:
        st.set_arith(arith)
        st.set(psi)
        e = st.expectation(xm, zm, cf)
    ref = _reference(psi, terms)
    size = sum(abs(_reference(psi, [t])) for t in terms)
    assert abs(e - float(ref)) <= tol * float(size), (e, ref)


@pytest.mark.parametrize("dtype,tol", [("c128", 1e-13), ("c64", 1e-12)])
def test_weights_beyond_a_float(dtype, tol):
    from paper_1604_06460_gb300 import qe
    psi = I.random_state(N, 9)
    if dtype == "c64":
        psi = psi.astype(np.complex64).astype(complex)
    for cf in ([1e-60, 3e-60], [1e60, 1e61], [1.0, 1e-50], [1e300, 1e-300]):
        for terms in ([(12, 0, cf[0]), (96, 1, cf[1])], [(12, 0, cf[0]), (0, 7, cf[1])]):
            xm, zm, w = (np.array(v, dtype=t) for v, t in zip(zip(*terms), (np.uint64, np.uint64, float)))
            with qe.State(N, dtype) as st:
                st.set(psi)
                e = st.expectation(xm, zm, w)
            assert abs(e - float(_reference(psi, terms))) <= tol * sum(cf)
