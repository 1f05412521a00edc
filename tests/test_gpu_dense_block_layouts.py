"""Dense blocks on tensor cores for every way a tile is moved: targets in any order
that leave out qubit 0, hold it, or hold the three (four, five) lowest, against
the oracle, within 4e-6 of sum_j |U_ij| max |psi| (the split operands' bound)."""
import numpy as np
import pytest

from oracle import statevec
from paper_1412_2293_gb300 import qs
from tests.test_gpu_dense_blocks import bound, rand_states, rand_unitary, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


@pytest.mark.parametrize("n,targets,members", [
    (10, (2, 0, 1), 3), (11, (0, 1, 2), 1), (12, (1, 0, 2, 3), 3), (12, (0, 9, 2, 1), 2), (11, (3, 1, 2, 0), 1),
    (12, (4, 2, 0, 1, 3), 3), (13, (2, 11, 0, 8, 1), 2), (13, (0, 1, 2, 3, 7), 2), (14, (13, 0, 2, 1, 3), 1),
    (12, (0, 5, 8), 3), (12, (6, 0, 1), 2), (13, (1, 0, 6, 9), 3), (13, (9, 1, 4, 0, 12), 2), (12, (1, 2, 3, 4, 5), 2),
    (20, (3, 0, 1, 2, 4), 4), (20, (19, 1, 0, 2), 4), (20, (2, 1, 0), 4),
])
def test_block_matches_oracle(n, targets, members):
    rng = np.random.default_rng(sum(targets) + n)
    U = rand_unitary(rng, 1 << len(targets))
    psi = rand_states(rng, members, n)
    got = run(n, members, targets, U, psi, qs.QS_C64)
    for b in range(members):
        want = statevec.apply_gate(psi[b], n, targets, U)
        assert np.abs(got[b] - want).max() <= 4e-6 * bound(U, psi[b])


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
@pytest.mark.parametrize("n,batch", [(1, 3), (2, 300), (5, 40), (9, 2), (10, 1), (14, 5), (16, 2), (18, 3)])
def test_small_noisy_gates_equal_the_planned_draws(n, batch, dtype):
    """Noisy gates whose draw shares their launch (small states) and those that do
    not, many members per block and many blocks per member, against the oracle."""
    from oracle import gates as ogates
    from oracle import philox
    rng = np.random.default_rng(n + batch)
    psi = rand_states(rng, batch, n)
    e, seed = 0.2, 99
    z = rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2))
    gates = [((0,), ogates.hadamard(), qs.QS_NOISE_ROTATION), ((n - 1,), np.linalg.qr(z)[0], qs.QS_NOISE_ROTATION),
             ((n // 2,), ogates.hadamard(), qs.QS_NOISE_PHASE), ((n - 1,), np.diag([1.0, 1j]), qs.QS_NOISE_PHASE)]
    if n > 1:
        gates += [((n - 1, 0), ogates.controlled_phase(0.7), qs.QS_NOISE_PHASE),
                  ((0, n - 1), np.diag(np.exp(1j * np.arange(4))), qs.QS_NOISE_PHASE),
                  ((0, n // 2 if n > 2 else 1), rand_unitary(rng, 4), qs.QS_NOISE_ROTATION)]
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_state(h, psi.ravel())
        qs.qs_set_trajectory_offset(h, 7)
        for g, (t, U, kind) in enumerate(gates):
            qs.qs_apply_noisy_gate(h, t, U, kind, e, seed, g)
        got = qs.qs_get_state(h).reshape(batch, -1)
    finally:
        qs.qs_destroy(h)
    for b in sorted(set([0, batch // 2, batch - 1])):
        want = psi[b]
        for g, (t, U, kind) in enumerate(gates):
            xa, xb = philox.normal_pair(seed, 7 + b, g)
            want = statevec.apply_gate(want, n, t, ogates.noisy_unitary(
                U, "phase" if kind == qs.QS_NOISE_PHASE else "rotation", e, xa, xb))
        # a gate rounds an amplitude a few times: 8 roundings per gate of the largest amplitude
        eps = 2.0 ** -24 if dtype == qs.QS_C64 else 2.0 ** -52
        np.testing.assert_allclose(got[b], want, rtol=0, atol=8 * len(gates) * eps * np.abs(want).max() * 2)
