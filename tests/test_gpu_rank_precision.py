"""Rounding of fixed-rank channels: what the trace of one that truncates nothing is
off by, over random factors, and that of a search whose cut amplifies it.

The rounding of the projection's matrices V and of the Kraus operators E is the same
for every row of L, so it does not average out.  A rounding of a random number is
0.42 u rms, u = 2^-53.  An entry of V takes two, and the trace, twice the relative
error of V, is carried by at least two of its entries: 2 sqrt(2) 0.42 u / sqrt(2) = 0.84 u.
E is a rounded square root times a rounded entry: 2 sqrt(2) 0.42 u = 1.2 u where the
oracle's roundings differ.  Together 1.5 u rms; 2 u allowed.  (A further rounding of
the eigenvectors, or their norms off by one, is 2.4 u.)"""
import numpy as np
import pytest

from oracle import circuits as ocirc
from oracle import fixed_rank as ofr
from oracle import gates as ogates
from paper_1412_2293_gb300 import circuits as pcirc
from paper_1412_2293_gb300 import inputs, qs

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


@pytest.mark.parametrize("n,e,marked", [(8, 0.0191, 141), (8, 0.0159, 52), (9, 0.0161, 240)])
def test_trace_of_a_truncated_search(n, e, marked):
    """Grover's search at rank 4, where the cut falls between eigenvalues hundreds of
    times closer to each other than to the largest: an error of the eigenvectors is
    divided by that gap.  The trace is allowed what 2 u a channel, all in one
    direction, come to on either side."""
    from paper_1412_2293_gb300 import build
    build.build()
    ops, r = inputs.grover_circuit(n, 9, marked), 4
    h = qs.qs_create(n, 1, r, qs.QS_FIXED_RANK, qs.QS_C128)
    try:
        qs.qs_set_basis_state(h, 0)
        pcirc.apply_ops(h, ops, e, 0)
        got = qs.qs_trace(h)[0]
    finally:
        qs.qs_destroy(h)
    want = ofr.trace(ocirc.run_fixed_rank(n, ops, 0, e, r))
    assert abs(got - want) <= 2 * 2 * 2.0 ** -53 * sum(o.noisy for o in ops)
