"""One fixed-rank channel on a random factor, for every form of its Kraus set and
the sizes where the kernels' splits change: one- and two-qubit, dense and
diagonal operators, explicit sets of up to eight, real and complex factors, up to
32 columns of L', members of uneven rank, close and tied eigenvalues.

Tolerance of L L^dagger: the Gram matrix carries about 10 roundings of 2^-53 of
its largest eigenvalue (the trace bounds it); a kept subspace moves by that over
the gap at the cut, which the factors below keep above 1e-4 of the trace:
4 x 10 x 2^-53 / 1e-4 < 1e-10; complex64 columns carry 2^-24 each, 1e-5 with the
factor of the gap (their cut is at a gap of 1e-1 or nothing is cut)."""
import numpy as np
import pytest

from oracle import fixed_rank as ofr
from oracle import gates as ogates
from oracle import relaxation as orx
from paper_1412_2293_gb300 import qs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def unitary(rng, D, real):
    z = rng.normal(size=(D, D)) + (0 if real else 1j) * rng.normal(size=(D, D))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


def factor(rng, n, m, real):
    L = rng.normal(size=(1 << n, m)) + (0 if real else 1j) * rng.normal(size=(1 << n, m))
    return L * 0.6 ** np.arange(m) / np.sqrt(1 << n)


def channel(kind, rng, real):
    """(k, gate arguments or None, Kraus set) of a form."""
    e = 0.3
    if kind == "rotation1":
        U = unitary(rng, 2, real)
        return 1, (U, qs.QS_NOISE_ROTATION, e), ogates.kraus_set(U, "rotation", e)
    if kind == "phase1":
        U = np.diag([1.0, -1.0 if real else np.exp(0.7j)])
        return 1, (U, qs.QS_NOISE_PHASE, e), ogates.kraus_set(U, "phase", e)
    if kind == "phase1_dense":
        U = unitary(rng, 2, real)
        return 1, (U, qs.QS_NOISE_PHASE, e), ogates.kraus_set(U, "phase", e)
    if kind == "phase2":
        U = np.diag(np.exp(1j * rng.uniform(0, 6, size=4)) * (0 if real else 1)) if not real else np.diag([1.0, 1, 1, -1])
        return 2, (U, qs.QS_NOISE_PHASE, e), ogates.kraus_set(U, "phase", e)
    if kind == "rotation2":
        U = unitary(rng, 4, real)
        return 2, (U, qs.QS_NOISE_ROTATION, e), ogates.kraus_set(U, "rotation", e)
    if kind == "relax":
        return 1, None, orx.relaxation_kraus(0.4, 2.0, 1.5)
    ks = [unitary(rng, 2, real) * np.sqrt(w) for w in np.arange(1, 9) / 36.0]      # eight unitaries
    return 1, None, ks


CASES = [  # kind, n, columns, rank, real
    ("rotation1", 1, 1, 1, True), ("rotation1", 4, 3, 5, False), ("rotation1", 9, 8, 8, True), ("rotation1", 9, 8, 8, False),
    ("rotation1", 11, 9, 12, True), ("rotation1", 12, 16, 16, False), ("rotation1", 15, 5, 7, True),
    ("phase1", 5, 3, 4, True), ("phase1", 10, 16, 16, False), ("phase1_dense", 6, 4, 8, False),
    ("phase2", 2, 2, 3, False), ("phase2", 6, 7, 7, True), ("phase2", 12, 8, 8, False), ("phase2", 13, 16, 16, False),
    ("rotation2", 5, 3, 6, True), ("rotation2", 8, 8, 8, False),
    ("relax", 7, 5, 10, False), ("relax", 8, 10, 10, True), ("eight", 7, 4, 9, False), ("eight", 6, 1, 8, True),
]


@pytest.mark.parametrize("kind,n,m,rank,real", CASES)
@pytest.mark.parametrize("dtype", [qs.QS_C128, qs.QS_C64])
def test_one_channel_matches_oracle(kind, n, m, rank, real, dtype):
    rng = np.random.default_rng(1000 * n + 10 * m + rank)
    k, gate, kraus = channel(kind, rng, real)
    targets = [int(t) for t in rng.choice(n, size=k, replace=False)]
    L = factor(rng, n, m, real)
    if dtype == qs.QS_C64:
        L = L.astype(np.complex64).astype(complex)
        rank = min(16, len(kraus) * m) if len(kraus) * m <= 16 else rank
    state = np.zeros((rank, 1 << n), dtype=complex)
    m = min(m, rank)
    L = L[:, :m]
    state[:m] = L.T
    h = qs.qs_create(n, 1, rank, qs.QS_FIXED_RANK, dtype)
    try:
        qs.qs_set_state(h, state.reshape(-1))
        qs.qs_set_rank_columns(h, m)
        if gate:
            qs.qs_apply_noisy_gate(h, targets, gate[0], gate[1], gate[2], 0, 0)
        else:
            qs.qs_apply_kraus(h, targets, kraus)
        cols = qs.qs_get_rank(h)
        got = qs.qs_get_state(h).reshape(rank, -1)[:cols].T
        tr = qs.qs_trace(h)[0]
    finally:
        qs.qs_destroy(h)
    want, lam = ofr.truncate(ofr.apply_kraus(L, n, targets, kraus), rank, False)
    lam = np.sort(lam)[::-1]
    assert cols == min(rank, len(kraus) * m)
    total = float(np.sum(np.abs(L) ** 2))
    if dtype == qs.QS_C64 and cols < len(kraus) * m:
        assert abs(tr - np.sum(np.abs(want) ** 2)) < 1e-5 * total       # the cut's gap is not wide enough for the matrix
        return
    tol = (1e-10 if dtype == qs.QS_C128 else 1e-5) * total
    rows = rng.choice(1 << n, size=min(1 << n, 64), replace=False)
    np.testing.assert_allclose(got[rows] @ got.conj().T, want[rows] @ want.conj().T, rtol=0, atol=tol)
    # the columns are eigenvectors: orthogonal, in descending order
    g = got.conj().T @ got
    assert np.abs(g - np.diag(np.diag(g))).max() < (1e-12 if dtype == qs.QS_C128 else 1e-5) * total
    np.testing.assert_allclose(np.diag(g).real, lam[:cols], rtol=0, atol=(1e-12 if dtype == qs.QS_C128 else 1e-5) * total)


@pytest.mark.parametrize("gap", [0.0, 1e-13, 3e-11, 2e-10, 1e-8, 1e-6])
def test_close_eigenvalues(gap):
    """Columns whose norms differ by `gap`: inside, at and outside a tie cluster,
    through the refinement and the FP64 Jacobi."""
    n, m = 8, 8
    rng = np.random.default_rng(5)
    q = np.linalg.qr(rng.normal(size=(1 << n, m)))[0]
    d = np.array([1.0, 0.02, 0.02 + gap, 0.02 + 2 * gap, 1e-4, 1e-4 + gap, 1e-9, 1e-9 * (1 + 1e-3)])
    L = q * np.sqrt(d) @ unitary(rng, m, True).T          # the eigenvalues are d, the columns mixed
    h = qs.qs_create(n, 1, 16, qs.QS_FIXED_RANK, qs.QS_C128)
    try:
        state = np.zeros((16, 1 << n), dtype=complex)
        state[:m] = L.T
        qs.qs_set_state(h, state.reshape(-1))
        qs.qs_set_rank_columns(h, m)
        qs.qs_apply_noisy_gate(h, (3,), ogates.hadamard(), qs.QS_NOISE_ROTATION, 0.01, 0, 0)
        got = qs.qs_get_state(h).reshape(16, -1).T
    finally:
        qs.qs_destroy(h)
    Lp = ofr.apply_kraus(L, n, (3,), ogates.kraus_set(ogates.hadamard(), "rotation", 0.01))
    np.testing.assert_allclose(got @ got.conj().T, Lp @ Lp.conj().T, rtol=0, atol=1e-14)


def test_uneven_members_equal_each_alone():
    n, ranks = 11, [1, 16, 3, 8]
    rng = np.random.default_rng(9)
    L = [factor(rng, n, r, False) for r in ranks]
    U = np.diag([1.0, 1.0, 1.0, np.exp(0.4j)])

    def run(members):
        R = max(ranks)
        h = qs.qs_create(n, len(members), R, qs.QS_FIXED_RANK, qs.QS_C128)
        try:
            qs.qs_set_member_ranks(h, [ranks[b] for b in members])
            s = np.zeros((len(members), R, 1 << n), dtype=complex)
            for i, b in enumerate(members):
                s[i, :1] = L[b][:, :1].T
            qs.qs_set_state(h, s.reshape(-1))
            qs.qs_set_rank_columns(h, 1)
            for g in range(5):
                qs.qs_apply_noisy_gate(h, (g,), ogates.hadamard(), qs.QS_NOISE_ROTATION, 0.2, 0, 0)
                qs.qs_apply_noisy_gate(h, (g, 10 - g), U, qs.QS_NOISE_PHASE, 0.3, 0, 0)
            return qs.qs_get_state(h).reshape(len(members), R, -1)
        finally:
            qs.qs_destroy(h)

    mixed = run([0, 1, 2, 3])
    for b in range(4):
        np.testing.assert_array_equal(mixed[b], run([b])[0])
