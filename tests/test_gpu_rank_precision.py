"""Rounding of fixed-rank channels that truncate nothing: what a channel's trace is
off by, over random factors.

The rounding of the projection's matrices V and of the Kraus operators E is the same
for every row of L, so it does not average out.  A rounding of a random number is
0.42 u rms, u = 2^-53.  An entry of V takes two, and the trace, twice the relative
error of V, is carried by at least two of its entries: 2 sqrt(2) 0.42 u / sqrt(2) = 0.84 u.
E is a rounded square root times a rounded entry: 2 sqrt(2) 0.42 u = 1.2 u where the
oracle's roundings differ.  Together 1.5 u rms; 2 u allowed.  (A further rounding of
the eigenvectors, or their norms off by one, is 2.4 u.)"""
import numpy as np
import pytest

from oracle import gates as ogates
from paper_1412_2293_gb300 import qs

pytestmark = pytest.mark.gpu


def test_trace_of_channels_without_truncation():
    from paper_1412_2293_gb300 import build
    build.build()
    n, off = 9, []
    for i in range(160):
        rng = np.random.default_rng(i)
        real, hadamard, m = bool(i % 2), bool(i // 2 % 2), int(rng.integers(1, 9))
        e = float(10 ** rng.uniform(-3, -0.7))
        q = np.linalg.qr(rng.normal(size=(1 << n, m)) + (0 if real else 1j) * rng.normal(size=(1 << n, m)))[0]
        d = float(rng.choice([0.6, 0.1, 0.01])) ** np.arange(m)
        mix = np.linalg.qr(rng.normal(size=(m, m)) + (0 if real else 1j) * rng.normal(size=(m, m)))[0]
        L = (q * np.sqrt(d / d.sum())) @ (mix if rng.random() < 0.5 else np.eye(m))
        if hadamard:
            U, noise, t = ogates.hadamard(), (qs.QS_NOISE_ROTATION, "rotation"), [int(rng.integers(n))]
        else:
            U = np.diag([1.0, 1.0, 1.0, -1.0 if real else np.exp(1j * rng.uniform(0, 6))]).astype(complex)
            noise, t = (qs.QS_NOISE_PHASE, "phase"), [int(x) for x in rng.choice(n, size=2, replace=False)]
        h = qs.qs_create(n, 1, 16, qs.QS_FIXED_RANK, qs.QS_C128)
        try:
            state = np.zeros((16, 1 << n), dtype=complex)
            state[:m] = L.T
            qs.qs_set_state(h, state.reshape(-1))
            qs.qs_set_rank_columns(h, m)
            qs.qs_apply_noisy_gate(h, t, U, noise[0], e, 0, 0)
            got = qs.qs_get_state(h)
        finally:
            qs.qs_destroy(h)
        # sum over rows of |sum_j E_aij l_j|^2 = sum_jk (E^H E)_jk <l_j, l_k>, in long double
        ll = L.astype(np.clongdouble).T
        E = [K.astype(np.clongdouble) for K in ogates.kraus_set(U, noise[1], e)]
        S = sum(K.conj().T @ K for K in E)
        rows = np.arange(1 << n)
        local = sum(((rows >> q) & 1) << j for j, q in enumerate(t))
        want = np.longdouble(0)
        for j in range(1 << len(t)):
            for k in range(1 << len(t)):
                if S[j, k] != 0:
                    a, b = ll[:, local == j], ll[:, local == k]
                    want += (S[j, k] * np.sum(a.conj() * b)).real
        off.append(float(np.sum(np.abs(got.astype(np.clongdouble)) ** 2) - want))
    assert np.sqrt(np.mean(np.square(off))) < 2 * 2.0 ** -53
