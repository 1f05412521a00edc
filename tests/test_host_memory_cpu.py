"""Host code of the library on a fake CUDA runtime (tests/fake_cudart.cc): the
device memory a handle and its plans take against the server's admission bound,
plans after an allocation failed, and what the autotuner picks from given times."""
import glob
import os
import subprocess
import sys

import pytest

from paper_1412_2293_gb300 import build

ROOT = build.ROOT


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """Path of the library linked against the fake runtime."""
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "obj", "*.o")))
    if not build.up_to_date() or len(objs) != len(build.sources()):
        build.build(force=True)
        objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "obj", "*.o")))
    out = str(tmp_path_factory.mktemp("fake") / "libqsim_fake.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", out, os.path.join(ROOT, "tests", "fake_cudart.cc"), *objs,
                    "-Wl,--no-undefined"], check=True, capture_output=True)
    return out


PRELUDE = """
import sys, ctypes as ct
sys.path.insert(0, {root!r})
from paper_1412_2293_gb300 import circuits, inputs, qs, server
qs.LIB_PATH = {lib!r}
L = qs.lib()
L.fake_device_bytes.restype = ct.c_size_t
L.fake_pinned_blocks.restype = ct.c_size_t
L.fake_pinned_calls.restype = ct.c_long
L.fake_fail_after.argtypes = [ct.c_long]
L.fake_cost.argtypes = [ct.c_char_p, ct.c_double]
def circuit(name, n, it):
    return circuits.to_gates(inputs.qft_circuit(n) if name == "qft" else inputs.grover_circuit(n, it, 1), per_member_flip=True)
"""


def run(lib, body):
    """The body in an interpreter of its own (a fault in host code ends that one only)."""
    r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, lib=lib) + body], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout[-2000:], r.stderr[-2000:])


def test_plan_stays_usable_after_a_window_width_found_no_memory(fake):
    run(fake, """
for fail in range(24):
    h = qs.qs_create(20, 4, 0, qs.QS_STATEVEC, qs.QS_C64)
    p = qs.qs_plan_create(h, circuit("qft", 20, 0))
    qs.qs_set_basis_state(h, 3)
    L.fake_fail_after(fail)
    try:
        qs.qs_plan_set_window(p, 12, h)
        L.fake_fail_after(-1)
        passes, launches = qs.qs_plan_info(p)
        assert passes == 2 and launches >= 5, (fail, passes, launches)
    except qs.QSError as err:
        assert err.status == qs.QS_ERR_OUT_OF_MEMORY, err
        assert qs.qs_plan_info(p) == (0, 0), (fail, qs.qs_plan_info(p))
        qs.qs_plan_set_window(p, 10, h)
        assert qs.qs_plan_info(p)[0] == 2
    qs.qs_plan_destroy(p)
    qs.qs_destroy(h)
assert L.fake_device_bytes() == 0
""")


# what the server runs: its smallest launch and larger ones, all widths, circuits of few and of thousands of passes
@pytest.mark.parametrize("name,n,it,members,m", [
    ("qft", 8, 0, 16, 10), ("qft", 13, 0, 64, 10), ("qft", 17, 0, 16, 10), ("qft", 20, 0, 256, 10), ("qft", 21, 0, 16, 11),
    ("qft", 24, 0, 16, 12), ("qft", 26, 0, 16, 10), ("grover", 10, 25, 16, 10), ("grover", 16, 201, 16, 10),
    ("grover", 12, 900, 16, 10), ("grover", 12, 900, 128, 10),
])
def test_admission_bound_covers_what_a_launch_allocates(fake, name, n, it, members, m):
    run(fake, f"""
name, n, it, B, m = {name!r}, {n}, {it}, {members}, {m}
h = qs.qs_create(n, B, 0, qs.QS_STATEVEC, qs.QS_C64)
p = qs.qs_plan_create(h, circuit(name, n, it))
qs.qs_plan_set_window(p, m, h)
qs.qs_set_member_noise(h, [0.01] * B, [1] * B, range(B), [1] * B)
qs.qs_set_basis_states(h, [0] * B)
used, bound = L.fake_device_bytes(), B * server.member_bytes(n)
assert used <= bound, (used / B, bound / B)
qs.qs_plan_destroy(p)
qs.qs_destroy(h)
assert L.fake_device_bytes() == 0
""")


# ms per pass by window width, from a start not yet written and from memory -> the width picked with a start pending
# and without: start times within 1/16 of each other are decided by the others
@pytest.mark.parametrize("start,memory,pending,loaded", [
    ((1.0, 0.98, 0.99), (3.5, 4.5, 5.0), 10, 10),
    ((1.0, 0.95, 0.99), (3.5, 4.5, 3.0), 12, 12),
    ((1.0, 0.9, 0.8), (3.5, 4.5, 5.0), 12, 10),
    ((1.0, 1.1, 1.2), (3.5, 3.0, 2.5), 10, 12),
])
def test_autotuned_width_from_a_pending_start(fake, start, memory, pending, loaded):
    run(fake, f"""
for m, s, d in zip((10, 11, 12), {start!r}, {memory!r}):
    L.fake_cost(b"Li%dELb1EE" % m, s)                 # the pass kernels, M = m, START
    L.fake_cost(b"Li%dELb0EE" % m, d)
h = qs.qs_create(24, 2, 0, qs.QS_STATEVEC, qs.QS_C64)
for start, want in ((True, {pending}), (False, {loaded})):
    p = qs.qs_plan_create(h, circuit("qft", 24, 0)[:1])   # one pass at every width
    if start:
        qs.qs_set_basis_state(h, 5)
    qs.qs_plan_autotune(p, 2, 0.01, 1, h)
    assert qs.qs_plan_get_window(p, h) == want, (want, qs.qs_plan_get_window(p, h))
    qs.qs_plan_run(p, 0.01, 1, 0, h)                  # no start is pending from here on
    qs.qs_plan_destroy(p)
qs.qs_destroy(h)
""")


def test_autotuner_times_the_fidelity_of_a_stored_reference(fake):
    run(fake, """
import numpy as np
L.fake_cost(b"k_outerIfLi4ELb0E", 1.0)                # k_outer without and with the fidelity
L.fake_cost(b"k_outerIfLi4ELb1E", 5.0)
for stored, want in ((False, 1.0), (True, 5.0)):
    h = qs.qs_create(20, 2, 0, qs.QS_STATEVEC, qs.QS_C64)
    if stored:
        qs.qs_set_reference(h, np.eye(1, 1 << 20, dtype=complex)[0])
    p = qs.qs_plan_create(h, circuit("qft", 20, 0))
    qs.qs_set_basis_state(h, 5)
    low, high = qs.qs_plan_autotune(p, 2, 0.01, 1, h)
    assert (low, high) == (want, 0.0), (low, high)
    qs.qs_plan_destroy(p)
    qs.qs_destroy(h)
""")
