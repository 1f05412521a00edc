"""Overlaps and norms from 20 qubits up, where a block takes four rounds of 4096
amplitudes: against FP64, and sums of rounds beyond FP32's range."""
import numpy as np
import pytest

from paper_1412_2293_gb300 import qs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


@pytest.mark.parametrize("dtype,tol", [(qs.QS_C64, 1e-6), (qs.QS_C128, 1e-13)])
@pytest.mark.parametrize("n,batch", [(20, 3), (21, 1)])
def test_overlaps_and_norms_in_rounds(n, batch, dtype, tol):
    rng = np.random.default_rng(n)
    N = 1 << n
    psi = rng.normal(size=(batch, N)) + 1j * rng.normal(size=(batch, N))
    psi /= np.linalg.norm(psi, axis=1, keepdims=True)
    ref = 0.8 * psi[0] + 0.3 * psi[-1][::-1]
    if dtype == qs.QS_C64:
        psi, ref = psi.astype(np.complex64).astype(complex), ref.astype(np.complex64).astype(complex)
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_state(h, psi.reshape(-1))
        f, t = qs.qs_fidelity(h, ref), qs.qs_trace(h)
    finally:
        qs.qs_destroy(h)
    np.testing.assert_allclose(f, np.abs(psi @ ref.conj()) ** 2, rtol=0, atol=2 * tol)
    np.testing.assert_allclose(t, np.sum(np.abs(psi) ** 2, axis=1), rtol=0, atol=tol)


def test_sums_of_rounds_beyond_fp32():
    """A thread's 16 products stay below 2^128, its four rounds do not: the sums of rounds are FP64's."""
    n, a = 20, 2.0 ** 61.5                                     # |a|^2 = 2^123: 2^127 a round
    N = 1 << n
    psi = np.full(N, a).astype(np.complex64).astype(complex)
    h = qs.qs_create(n, 1, 0, qs.QS_STATEVEC, qs.QS_C64)
    try:
        qs.qs_set_state(h, psi)
        f, t = qs.qs_fidelity(h, psi)[0], qs.qs_trace(h)[0]
    finally:
        qs.qs_destroy(h)
    want = N * psi[0].real ** 2
    assert abs(t / want - 1) <= 2.0 ** -20 and abs(f / want ** 2 - 1) <= 2.0 ** -19
