"""Reductions at the sizes where their splits change: one warp or one block per
result (64 partials), chunks of 4096 amplitudes, groups of columns, the
Hermitian and the full expectation of a density matrix."""
import numpy as np
import pytest

from paper_1412_2293_gb300 import qs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def random_state(rng, shape):
    s = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    return s / np.sqrt(np.sum(np.abs(s) ** 2, axis=-1, keepdims=True))


@pytest.mark.parametrize("dtype,tol", [(qs.QS_C64, 1e-6), (qs.QS_C128, 1e-13)])
@pytest.mark.parametrize("n,batch", [(1, 3), (11, 2), (12, 5), (13, 1), (18, 2), (19, 1)])
def test_statevector_overlaps_and_norms(n, batch, dtype, tol):
    rng = np.random.default_rng(100 * n + batch)
    psi = random_state(rng, (batch, 1 << n))
    ref = random_state(rng, (1 << n,)) + 0.5 * psi[0]
    if dtype == qs.QS_C64:
        psi, ref = psi.astype(np.complex64).astype(complex), ref.astype(np.complex64).astype(complex)
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_state(h, psi.reshape(-1))
        f, t = qs.qs_fidelity(h, ref), qs.qs_trace(h)
    finally:
        qs.qs_destroy(h)
    np.testing.assert_allclose(f, np.abs(psi @ ref.conj()) ** 2, rtol=0, atol=tol * 2)
    np.testing.assert_allclose(t, np.sum(np.abs(psi) ** 2, axis=1), rtol=0, atol=tol)


@pytest.mark.parametrize("n,rank,batch", [(3, 1, 2), (12, 5, 3), (13, 8, 1), (14, 16, 2)])
def test_fixed_rank_group_sums(n, rank, batch):
    rng = np.random.default_rng(n * rank)
    L = random_state(rng, (batch, rank, 1 << n))
    ref = random_state(rng, (1 << n,)) + L[0, 0]
    h = qs.qs_create(n, batch, rank, qs.QS_FIXED_RANK, qs.QS_C128)
    try:
        qs.qs_set_state(h, L.reshape(-1))
        qs.qs_set_rank_columns(h, rank)
        f, t = qs.qs_fidelity(h, ref), qs.qs_trace(h)
    finally:
        qs.qs_destroy(h)
    np.testing.assert_allclose(f, np.sum(np.abs(L @ ref.conj()) ** 2, axis=1), rtol=1e-13)
    np.testing.assert_allclose(t, np.full(batch, float(rank)), rtol=1e-13)


@pytest.mark.parametrize("dtype,tol", [(qs.QS_C64, 1e-12), (qs.QS_C128, 1e-13)])
@pytest.mark.parametrize("n", [1, 4, 8, 9])
@pytest.mark.parametrize("hermitian", [True, False])
def test_density_expectation(n, hermitian, dtype, tol):
    """The sum itself carries at least 48 bits in either precision (the
    amplitudes given are exact in the handle's precision)."""
    rng = np.random.default_rng(n)
    N = 1 << n
    rho = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    if hermitian:
        rho = rho + rho.conj().T
    rho /= np.linalg.norm(rho)
    phi = random_state(rng, (N,))
    if dtype == qs.QS_C64:
        rho, phi = rho.astype(np.complex64).astype(complex), phi.astype(np.complex64).astype(complex)
    h = qs.qs_create(n, 1, 0, qs.QS_DENSITY, dtype)
    try:
        qs.qs_set_state(h, rho.reshape(-1))
        got = qs.qs_fidelity(h, phi)[0]
    finally:
        qs.qs_destroy(h)
    want = np.vdot(phi, rho @ phi).real
    assert abs(got - want) <= tol * np.sum(np.abs(phi[:, None] * rho * phi[None, :]))
