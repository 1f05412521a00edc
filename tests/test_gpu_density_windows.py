"""Density plans run as window sweeps (n >= 8 in complex64, n >= 11 in complex128)
against the same channels one by one, and small ones against the oracle: windows
low, high and scattered, real channels of both forms, runs of diagonal channels
before, between and after, plans that break the windows, a matrix that is not
Hermitian."""
import numpy as np
import pytest

from oracle import density as odm
from oracle import gates as ogates
from paper_1412_2293_gb300 import circuits as pcirc
from paper_1412_2293_gb300 import inputs, qs

pytestmark = pytest.mark.gpu
SEED = inputs.DEFAULT_SEED


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def ry(t):
    return np.array([[np.cos(t), -np.sin(t)], [np.sin(t), np.cos(t)]])


def gates(kind, n, rng):
    """(gate, apply arguments) pairs."""
    out = []

    def one(q, U, noisy, noise=qs.QS_NOISE_ROTATION):
        out.append(((int(q),), np.asarray(U, dtype=complex), noisy, noise))

    def cp(j, k, noisy=True):
        out.append(((int(k), int(j)), ogates.controlled_phase(float(rng.uniform(0, 6))), noisy, qs.QS_NOISE_PHASE))

    if kind == "qft":
        for j in range(n - 1, -1, -1):
            one(j, ogates.hadamard(), True)
            for k in range(j - 1, -1, -1):
                cp(j, k)
        return out
    order = {"low": [0, 1, 2, 3, 4, 5, 0, 2], "high": list(range(n - 1, n - 7, -1)), "scattered": list(rng.permutation(n))}[
        "scattered" if kind in ("scattered", "breaks") else kind]
    cp(order[0], order[-1] if order[-1] != order[0] else (order[0] + 1) % n)      # a diagonal run first
    for i, q in enumerate(order):
        r = i % 4
        if r == 0:
            one(q, ogates.hadamard(), True)
        elif r == 1:
            one(q, ry(0.3 + i), True)
        elif r == 2:
            one(q, ry(1.1 * i), False)
        else:
            one(q, ogates.hadamard(), True, qs.QS_NOISE_PHASE)
        for _ in range(int(rng.integers(0, 3))):
            j, k = rng.choice(n, size=2, replace=False)
            cp(j, k, bool(rng.random() < 0.7))
        if kind == "breaks" and i % 3 == 2:
            q2 = int((q + 1) % n)
            z = rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2))
            one(q2, np.linalg.qr(z)[0], True)            # complex: its own sweep
    return out


@pytest.mark.parametrize("kind", ["qft", "low", "high", "scattered", "breaks"])
@pytest.mark.parametrize("n,dtype", [(8, qs.QS_C64), (9, qs.QS_C64), (10, qs.QS_C64), (11, qs.QS_C64), (11, qs.QS_C128),
                                     (12, qs.QS_C128)])
@pytest.mark.parametrize("hermitian", [True, False])
def test_plan_equals_channels_one_by_one(kind, n, dtype, hermitian):
    """Every entry goes through the same products in another order, a few roundings
    per channel: within 8 channels x 2^-24 (2^-53) of the largest entry."""
    if not hermitian and n > 10:
        pytest.skip("the sweeps of a general matrix do not depend on n")
    rng = np.random.default_rng(n)
    gs = gates(kind, n, rng)
    e = 0.1
    N = 1 << n
    v = rng.normal(size=(N, 2)) + 1j * rng.normal(size=(N, 2))
    rho = v @ v.conj().T
    rho = (rho + rho.conj().T) / (2 * np.trace(rho).real)
    if not hermitian:
        rho[0, 1] += 0.01
    if dtype == qs.QS_C64:
        rho = rho.astype(np.complex64).astype(complex)
    h = qs.qs_create(n, 1, 0, qs.QS_DENSITY, dtype)
    try:
        p = qs.qs_plan_create(h, [qs.make_gate(t, U, noisy=b, noise=z) for t, U, b, z in gs])
        if kind == "qft":
            assert qs.qs_plan_info(p)[0] <= (n + 3) // 4 if dtype == qs.QS_C64 else qs.qs_plan_info(p)[0] <= 3
        qs.qs_set_state(h, rho.reshape(-1))
        qs.qs_plan_run(p, e, SEED, 0, h)
        got = qs.qs_get_state(h).reshape(N, N)
        qs.qs_plan_destroy(p)
        qs.qs_set_state(h, rho.reshape(-1))
        for g, (t, U, b, z) in enumerate(gs):
            if b:
                qs.qs_apply_noisy_gate(h, t, U, z, e, SEED, g)
            else:
                qs.qs_apply_gate(h, t, U)
        want = qs.qs_get_state(h).reshape(N, N)
    finally:
        qs.qs_destroy(h)
    eps = 2.0 ** -24 if dtype == qs.QS_C64 else 2.0 ** -53
    np.testing.assert_allclose(got, want, rtol=0, atol=8 * len(gs) * eps * np.abs(want).max())
    if hermitian and kind != "breaks":
        np.testing.assert_array_equal(got, got.conj().T)


@pytest.mark.parametrize("kind", ["qft", "scattered"])
def test_complex64_windows_match_oracle(kind):
    n, e = 8, 0.2
    rng = np.random.default_rng(77)
    gs = gates(kind, n, rng)
    rho = odm.pure(np.eye(1 << n, dtype=complex)[37])
    h = qs.qs_create(n, 1, 0, qs.QS_DENSITY, qs.QS_C64)
    try:
        qs.qs_set_basis_state(h, 37)
        p = qs.qs_plan_create(h, [qs.make_gate(t, U, noisy=b, noise=z) for t, U, b, z in gs])
        qs.qs_plan_run(p, e, SEED, 0, h)
        got = qs.qs_get_state(h).reshape(1 << n, -1)
        qs.qs_plan_destroy(p)
    finally:
        qs.qs_destroy(h)
    for t, U, b, z in gs:
        ks = ogates.kraus_set(U, "phase" if z == qs.QS_NOISE_PHASE else "rotation", e) if b else [U]
        rho = odm.apply_channel(rho, n, t, ks)
    np.testing.assert_allclose(got, rho, rtol=0, atol=8 * len(gs) * 2.0 ** -24 * np.abs(rho).max())
