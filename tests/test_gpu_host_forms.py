"""Forms of the host path that few callers meet, bit for bit against the usual ones:
uploads and results of batches too large for the pinned staging block, plans whose
passes share one parameter block, members' noise changed between one-launch gates."""
import numpy as np
import pytest

from paper_1412_2293_gb300 import circuits as pcirc
from paper_1412_2293_gb300 import inputs, qs

pytestmark = pytest.mark.gpu
H = pcirc.hadamard()


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    return qs.lib()


def members(count, n):
    """Noise levels, keys, counters and starts of members 0.. (the same whatever the count)."""
    b = np.arange(count, dtype=np.uint64)
    return 0.01 + 1e-6 * b, 5 + b % 7, b * 3, (b * 5 + 1) % (1 << n)


def test_batch_beyond_the_pinned_block():
    n = 3

    def run(count):
        h = qs.qs_create(n, count, 0, qs.QS_STATEVEC, qs.QS_C64)
        try:
            out = []
            for turn in range(2):                     # the second upload replaces the first
                e, seed, traj, xs = members(count, n)
                qs.qs_set_member_noise(h, e + turn, seed, traj)
                qs.qs_set_basis_states(h, (xs + turn) % 8)
                for q in range(n):
                    qs.qs_apply_noisy_gate(h, (q,), H, qs.QS_NOISE_ROTATION, 0.0, 0, q)
                out.append((qs.qs_fidelity(h, None, 6), qs.qs_get_state(h).reshape(count, -1)))
            return out
        finally:
            qs.qs_destroy(h)

    few, many = run(40000), run(90000)                # 6 doubles a member: the block ends at 2^19
    for (f, s), (F, S) in zip(few, many):
        np.testing.assert_array_equal(f, F[:40000])
        np.testing.assert_array_equal(s, S[:40000])
        assert np.abs(F - np.abs(S[:, 6]) ** 2).max() < 1e-6


def test_passes_that_share_a_parameter_block():
    n = 16
    gates = pcirc.to_gates(inputs.grover_circuit(n, 800, 77))
    got, kernels = [], []
    for count in (2, 16):                             # 16 members' blocks of all passes are over the bound
        h = qs.qs_create(n, count, 0, qs.QS_STATEVEC, qs.QS_C64)
        try:
            p = qs.qs_plan_create(h, gates)
            passes, launches = qs.qs_plan_info(p, h)
            kernels.append(launches)
            qs.qs_set_basis_state(h, 0)
            qs.qs_plan_run(p, 0.001, 11, 0, h)
            got.append(qs.qs_get_state_range(h, 0, 2 << n))
            qs.qs_plan_destroy(p)
        finally:
            qs.qs_destroy(h)
    assert kernels[1] - kernels[0] == passes - 1      # a parameter launch per pass against one
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("dtype", [qs.QS_C64, qs.QS_C128])
def test_member_noise_changed_between_gates(dtype):
    n, count, turns = 5, 6, 24
    cp = pcirc.controlled_phase(0.7)

    def gate(h, g, e, seed):
        if g % 3:
            qs.qs_apply_noisy_gate(h, (g % n,), H, qs.QS_NOISE_ROTATION, e, seed, g)
        else:
            qs.qs_apply_noisy_gate(h, (g % n, (g + 2) % n), cp, qs.QS_NOISE_PHASE, e, seed, g)

    def noise(g):
        e, seed, traj, _ = members(count, n)
        return e * (1 + g), seed + g, traj + 2 * g

    h = qs.qs_create(n, count, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_basis_state(h, 3)
        for g in range(turns):
            qs.qs_set_member_noise(h, *noise(g))
            gate(h, g, 0.0, 0)
        mixed = qs.qs_get_state(h).reshape(count, -1)
    finally:
        qs.qs_destroy(h)
    for b in range(count):
        h = qs.qs_create(n, 1, 0, qs.QS_STATEVEC, dtype)
        try:
            qs.qs_set_basis_state(h, 3)
            for g in range(turns):
                e, seed, traj = (x[b] for x in noise(g))
                qs.qs_set_trajectory_offset(h, int(traj))
                gate(h, g, float(e), int(seed))
            np.testing.assert_array_equal(qs.qs_get_state(h), mixed[b])
        finally:
            qs.qs_destroy(h)
