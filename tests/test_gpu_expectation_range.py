"""<phi|rho|phi> of a complex64 density matrix carries FP64's bits at every
magnitude its entries can have: products beyond FP32's range, remainders below
it, sums that cancel, rows of zeros beside tiny ones."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1412_2293_gb300 import qs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def expectation(rho, phi):
    n = int(np.log2(len(phi)))
    h = qs.qs_create(n, 1, 0, qs.QS_DENSITY, qs.QS_C64)
    try:
        qs.qs_set_state(h, rho.astype(complex).reshape(-1))
        qs.qs_set_reference(h, phi.astype(complex))
        return qs.qs_fidelity_stored(h)[0]
    finally:
        qs.qs_destroy(h)


# rho and phi scales as powers of two: ordinary; products above 2^128; products whose remainders (2^-24 of them) fall
# below FP32's smallest number; whole products below it
@pytest.mark.parametrize("rho_exp,phi_exp", [(0, 0), (80, 50), (20, 30), (-40, -60), (-70, -70), (-100, -80)])
@pytest.mark.parametrize("hermitian", [True, False])
@pytest.mark.parametrize("n", [3, 9])
def test_expectation_at_every_magnitude(n, hermitian, rho_exp, phi_exp):
    rng = np.random.default_rng([n, rho_exp + 200, phi_exp + 200])
    N = 1 << n
    rho = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    if hermitian:
        rho = rho + rho.conj().T
    phi = rng.normal(size=N) + 1j * rng.normal(size=N)
    rho[:, 2] = 0
    rho[2, :] = 0
    rho = (rho * 2.0 ** rho_exp).astype(np.complex64)
    phi = (phi * 2.0 ** phi_exp).astype(np.complex64)
    if hermitian:
        rho = np.triu(rho, 1) + np.triu(rho, 1).conj().T + np.diag(rho.diagonal().real)
    got = expectation(rho, phi)
    r, f = rho.astype(complex) * 2.0 ** -rho_exp, phi.astype(complex) * 2.0 ** -phi_exp
    scale = 2.0 ** (rho_exp + 2 * phi_exp)
    want = np.vdot(f, r @ f).real
    # FP64 sums of exact products: a thread's N / 256 entries, 8 + 3 + 11 levels of sums, and numpy's own
    terms = np.abs(f) @ np.abs(r) @ np.abs(f)
    assert abs(got / scale - want) <= 64 * 2.0 ** -53 * terms


def test_expectation_of_entries_that_cancel():
    """Row sums far below their terms: FP64's error is a part of the terms, 2^-53, not 2^-48."""
    n, N = 6, 64
    rng = np.random.default_rng(5)
    phi = np.ones(N, dtype=np.complex64)
    rho = np.zeros((N, N), dtype=np.complex64)
    big = (rng.integers(1 << 23, 1 << 24, size=(N, N // 2)) * 2.0 ** 20).astype(np.float32)
    small = rng.integers(1, 1 << 10, size=(N, N // 2)).astype(np.float32)
    rho[:, 0::2] = big
    rho[:, 1::2] = -big
    rho[:, 0] = small[:, 0]
    rho[:, 1] = small[:, 1]
    want = sum((Fraction(float(v)) for v in rho.real.reshape(-1)), Fraction(0))
    got = expectation(rho, phi)
    assert abs(got - float(want)) <= 64 * 2.0 ** -53 * float(np.abs(rho.astype(complex)).sum())
