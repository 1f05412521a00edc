"""Runs of a plan from basis states, which follow the support of the state (only
the tiles and amplitudes that can differ from zero until every qubit has had a
dense gate, the last of those passes as an outer product where its tiles differ
by one amplitude), against the same plan from the same start written to memory.

Both apply the same gates in FP32 (FP64) in another order of products; a circuit
of G gates rounds an amplitude at most a few times per gate, so they agree
within 4 G 2^-24 (2^-53) of the rms amplitude, taken element by element."""
import numpy as np
import pytest

from paper_1412_2293_gb300 import circuits as pcirc
from paper_1412_2293_gb300 import inputs, qs
from paper_1412_2293_gb300.inputs import Op

pytestmark = pytest.mark.gpu
SEED = inputs.DEFAULT_SEED


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def ascending(n):
    """The QFT's gates from the lowest qubit up: low window first, out terms in the last pass."""
    ops = []
    for j in range(n):
        for k in range(j):
            ops.append(Op("CP", (j, k), theta=3.0 / (1 << (j - k)), noisy=True))
        ops.append(Op("H", (j,), noisy=True))
    return ops


def scattered(n, rng, flips):
    ops = [Op("H", (int(q),), noisy=True) for q in rng.permutation(n)]
    for _ in range(40):
        r = rng.random()
        if r < 0.4:
            ops.append(Op("H", (int(rng.integers(n)),), noisy=True))
        elif r < 0.9 or not flips:
            j, k = rng.choice(n, size=2, replace=False)
            ops.append(Op("CP", (int(max(j, k)), int(min(j, k))), theta=float(rng.uniform(0, 6)), noisy=True))
        else:
            ops.append(Op("FLIP", index=int(rng.integers(1 << n))))
    return ops


def circuit(kind, n, rng):
    if kind == "qft":
        return inputs.qft_circuit(n)
    if kind == "ascending":
        return ascending(n)
    if kind == "grover":
        return inputs.grover_circuit(n, 2, int(rng.integers(1, 1 << n)))
    if kind == "top_only":                                # never touches the low qubits
        return [Op("H", (q,), noisy=True) for q in range(n - 4, n)] + [Op("CP", (n - 1, 0), theta=0.4, noisy=True)]
    if kind == "late":                                    # one qubit has its first dense gate in the last pass
        return [o for o in inputs.qft_circuit(n) if o.qubits[0] != n - 1] + [Op("H", (n - 1,), noisy=True)]
    return scattered(n, rng, kind == "flips")


CASES = [  # circuit, n, members, dtype, window
    ("qft", 11, 2100, qs.QS_C64, 10), ("qft", 13, 520, qs.QS_C64, 10), ("qft", 13, 7, qs.QS_C64, 10),
    ("qft", 15, 130, qs.QS_C64, 11), ("qft", 16, 65, qs.QS_C64, 12), ("qft", 20, 5, qs.QS_C64, 10),
    ("qft", 21, 3, qs.QS_C64, 10), ("qft", 22, 1, qs.QS_C64, 11), ("qft", 22, 2, qs.QS_C64, 12),
    ("qft", 11, 130, qs.QS_C128, 10), ("qft", 14, 17, qs.QS_C128, 10), ("qft", 14, 3, qs.QS_C128, 10),
    ("ascending", 13, 6, qs.QS_C64, 10), ("ascending", 20, 3, qs.QS_C64, 10), ("ascending", 21, 2, qs.QS_C64, 12),
    ("ascending", 13, 3, qs.QS_C128, 10),
    ("grover", 12, 1030, qs.QS_C64, 10), ("grover", 16, 70, qs.QS_C64, 10), ("grover", 16, 5, qs.QS_C64, 12),
    ("random", 13, 5, qs.QS_C64, 10), ("random", 18, 17, qs.QS_C64, 10), ("random", 21, 2, qs.QS_C64, 11),
    ("flips", 14, 4, qs.QS_C64, 10), ("flips", 20, 4, qs.QS_C64, 10), ("flips", 13, 4, qs.QS_C128, 10),
    ("top_only", 15, 3, qs.QS_C64, 10), ("late", 14, 300, qs.QS_C64, 10), ("late", 21, 2, qs.QS_C64, 10),
    ("qft", 10, 3, qs.QS_C64, 10),
]


@pytest.mark.parametrize("kind,n,batch,dtype,m", CASES)
@pytest.mark.parametrize("per_member", [False, True])
def test_run_from_a_basis_start_equals_the_run_from_memory(kind, n, batch, dtype, m, per_member):
    rng = np.random.default_rng(n * 100 + batch)
    ops = circuit(kind, n, rng)
    e = 0.05
    xs = rng.integers(1 << n, size=batch) if per_member else np.full(batch, rng.integers(1 << n))
    ref = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    ref /= np.linalg.norm(ref)
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        # whatever is in memory before the run must not matter
        junk = np.full((min(batch, 2), 1 << n), np.nan + 1j * np.nan)
        if batch << n <= 1 << 22:
            qs.qs_set_state(h, np.full(batch << n, np.nan + 1j * np.nan))
        del junk
        qs.qs_set_reference(h, ref)
        p = qs.qs_plan_create(h, pcirc.to_gates(ops))
        if m != 10:
            qs.qs_plan_set_window(p, m)

        def start():
            if per_member:
                qs.qs_set_basis_states(h, xs)
            else:
                qs.qs_set_basis_state(h, int(xs[0]))

        pick = sorted(set([0, batch // 2, batch - 1]))

        def state():
            return np.stack([qs.qs_get_state_range(h, b << n, 1 << n) for b in pick])

        start()
        f_got = qs.qs_plan_run_fidelity(p, e, SEED, 3, h)
        got = state()
        start()
        qs.qs_plan_run(p, e, SEED, 3, h)                  # the same without the reduction
        again = state()
        start()
        qs.qs_apply_phase_flip(h, 0)                      # writes the start to memory
        qs.qs_apply_phase_flip(h, 0)
        f_want = qs.qs_plan_run_fidelity(p, e, SEED, 3, h)
        want = state()
        tr = qs.qs_trace(h)
        qs.qs_plan_destroy(p)
    finally:
        qs.qs_destroy(h)
    np.testing.assert_array_equal(got, again)
    eps = 2.0 ** -24 if dtype == qs.QS_C64 else 2.0 ** -53
    tol = 4 * max(len(ops), 10) * eps
    for g, w in zip(got, want):
        nz = np.abs(w[np.abs(w) > 0])
        np.testing.assert_allclose(g, w, rtol=0, atol=tol * (np.sqrt(np.mean(nz ** 2)) + np.abs(w).max()))
    # overlaps: 2^n products of a random reference, the same relative bound on the norm product
    np.testing.assert_allclose(f_got, f_want, rtol=0, atol=2 * tol)
    np.testing.assert_allclose(tr, 1.0, atol=2 * tol)


@pytest.mark.parametrize("n,batch,dtype,m", [(10, 3, qs.QS_C64, 10), (12, 5, qs.QS_C64, 10), (14, 2, qs.QS_C64, 11),
                                             (16, 3, qs.QS_C64, 12), (20, 2, qs.QS_C64, 10), (22, 1, qs.QS_C64, 10),
                                             (12, 2, qs.QS_C128, 10), (16, 2, qs.QS_C128, 10)])
@pytest.mark.parametrize("kind", ["system", "random"])
def test_run_from_the_entangled_start_equals_the_run_from_memory(n, batch, dtype, m, kind):
    rng = np.random.default_rng(n)
    ops = inputs.qft_circuit(n // 2) if kind == "system" else scattered(n, rng, True)
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_maximally_entangled(h)
        qs.qs_set_reference_from(h, h, batch - 1)
        p = qs.qs_plan_create(h, pcirc.to_gates(ops))
        if m != 10:
            qs.qs_plan_set_window(p, m)
        qs.qs_set_state(h, np.full(batch << n, np.nan + 1j * np.nan))      # memory must not matter
        qs.qs_set_maximally_entangled(h)
        f_got = qs.qs_plan_run_fidelity(p, 0.05, SEED, 3, h)
        got = qs.qs_get_state(h)
        qs.qs_set_maximally_entangled(h)
        qs.qs_apply_phase_flip(h, 0)                      # writes the start to memory
        qs.qs_apply_phase_flip(h, 0)
        f_want = qs.qs_plan_run_fidelity(p, 0.05, SEED, 3, h)
        want = qs.qs_get_state(h)
        qs.qs_plan_destroy(p)
    finally:
        qs.qs_destroy(h)
    # created and loaded registers hold the same bits, and the same gates follow
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(f_got, f_want)


@pytest.mark.parametrize("n", [12, 20])
def test_autotune_keeps_default_of_passes_without_a_choice(n):
    """Every pass of the QFT from a pending basis start has one form, so timing
    configurations there chooses nothing."""
    h = qs.qs_create(n, 2, 0, qs.QS_STATEVEC, qs.QS_C64)
    p = qs.qs_plan_create(h, pcirc.to_gates(inputs.qft_circuit(n)))
    try:
        qs.qs_set_basis_state(h, 3)
        qs.qs_plan_autotune(p, 1, 0.01, SEED, h)
        assert tuple(qs.qs_plan_get_config(p, h)) == ((2, 1) if qs.qs_plan_get_window(p, h) == 10 else (0, 0))
    finally:
        qs.qs_plan_destroy(p)
        qs.qs_destroy(h)
