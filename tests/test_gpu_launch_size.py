"""A trajectory's amplitudes and fidelity do not depend on how many members share
its launch: the same trajectories in small and large batches, bit by bit, on both
sides of the sizes where a run from a basis state ends in the outer product, and
in launches whose outer product takes its members in several turns."""
import numpy as np
import pytest

from paper_1412_2293_gb300 import circuits as pcirc
from paper_1412_2293_gb300 import inputs, qs

pytestmark = pytest.mark.gpu
SEED = inputs.DEFAULT_SEED


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1412_2293_gb300 import build
    build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return qs.lib()


def run_qft(n, batch, dtype, m, per_member, ref, take):
    """Fidelities and the first and last of `take` members of a planned QFT."""
    h = qs.qs_create(n, batch, 0, qs.QS_STATEVEC, dtype)
    try:
        qs.qs_set_reference(h, ref)
        p = qs.qs_plan_create(h, pcirc.to_gates(inputs.qft_circuit(n)))
        qs.qs_plan_set_window(p, m, h)
        if per_member:
            qs.qs_set_basis_states(h, [(37 * b + 5) % (1 << n) for b in range(batch)])
        else:
            qs.qs_set_basis_state(h, 5)
        f = qs.qs_plan_run_fidelity(p, 0.02, SEED, 0, h)
        qs.qs_plan_destroy(p)
        N = 1 << n
        return f[:take], qs.qs_get_state_range(h, 0, N), qs.qs_get_state_range(h, (take - 1) * N, N), f, \
            qs.qs_get_state_range(h, (batch - 1) * N, N)
    finally:
        qs.qs_destroy(h)


@pytest.mark.parametrize("n,small,large,dtype,m,per_member", [
    (13, 64, 512, qs.QS_C64, 10, True),
    (16, 2, 65, qs.QS_C64, 10, True),
    (17, 1, 33, qs.QS_C64, 10, False),
    (17, 3, 514, qs.QS_C64, 12, True),       # window states of 513 members and more: two turns
    (18, 2, 20, qs.QS_C64, 11, False),
    (12, 2, 300, qs.QS_C128, 10, False),
    (13, 2, 33, qs.QS_C128, 10, False),
    (14, 3, 1025, qs.QS_C128, 10, True),     # two turns
    (15, 2, 9, qs.QS_C128, 10, True),
])
def test_trajectories_same_in_small_and_large_launches(n, small, large, dtype, m, per_member):
    rng = np.random.default_rng(n)
    ref = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    ref /= np.linalg.norm(ref)
    a = run_qft(n, small, dtype, m, per_member, ref, small)
    b = run_qft(n, large, dtype, m, per_member, ref, small)
    for x, y, what in zip(a, b, ("fidelities", "first member", "last shared member")):
        np.testing.assert_array_equal(x, y, err_msg=what)
    # the members of the later turns too: the last one's fidelity is that of its state
    tol = 1e-5 if dtype == qs.QS_C64 else 1e-12
    assert abs(b[3][-1] - abs(np.vdot(ref, b[4])) ** 2) <= tol
    assert abs(np.linalg.norm(b[4]) - 1.0) <= tol


def test_server_job_same_in_a_small_and_a_large_launch():
    from paper_1412_2293_gb300.server import GpuExecutor, JobState, Slice, Unit, member_bytes
    n, count = 13, 64
    job = inputs.Job(0, 0.0, "qft", n, "statevec", count, 0, 1e-2, 77, 0)
    ex = GpuExecutor(workers=1, cache_bytes=0)
    try:
        got = []
        for members in (64, 512):
            u = Unit("mc", ("mc", "qft", n, 0), [Slice(0, 0, count)], members, members * member_bytes(n))
            got.append(ex.run(0, u, {0: JobState(job, 0.0)})[0])
            ex.release_job(0)
        np.testing.assert_array_equal(got[0], got[1])
    finally:
        ex.close()
