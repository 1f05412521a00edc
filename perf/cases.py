"""Performance cases: what a user of the simulator has it do, through qs.py.

Six kinds of pass, each as a program that estimates fidelities runs it:

gates    a noisy circuit issued gate by gate through the single-gate calls
         (no plan, no batching), the state read back: the plain form of the
         method, bound by calls and launches at small sizes.
mc       Monte Carlo trajectories of a planned noisy circuit from basis
         states.  jobs = 0: one job, qs_plan_run_fidelity against a stored
         reference; jobs > 0: what the server does with a launch -- the
         members' own noise and starts uploaded, one plan run, every job's
         fidelities against its own reference.
choi     trajectories of a circuit on the system half of the maximally
         entangled state (relative states): the planned passes on a state
         that is dense from the start.
rank     fixed-rank factors of a batch of jobs with their own ranks and noise
         levels, a planned circuit, then fidelity and trace.
density  the exact density matrix through a planned circuit, T1/T2 relaxation
         of every qubit where asked for, then fidelity and trace.
blocks   dense blocks of 3 to 5 qubits with a noisy Hadamard after each, gate
         by gate on a batch of trajectories, then the fidelities.

complex64 results are returned in single precision (what the arithmetic
carries), complex128 results in double.
"""
import math

import numpy as np
import torch

from paper_1412_2293_gb300 import circuits, inputs, qs
from paper_1412_2293_gb300.inputs import Op

DTYPES = {"c64": qs.QS_C64, "c128": qs.QS_C128}
ESIZE = {"c64": 8, "c128": 16}


def listed():
    return [
        # one trajectory of the plain method, gate by gate, complex128: 55 calls and a read-back
        {"name": "gates_qft_n10_c128", "kind": "gates", "circuit": "qft", "iterations": 0, "n": 10, "batch": 1, "dtype": "c128", "e": 0.01},
        # the smallest launch of the serving stream: two jobs of 32 trajectories share one
        {"name": "serve_qft_n13_c64_t64", "kind": "mc", "circuit": "qft", "iterations": 0, "n": 13, "batch": 64, "dtype": "c64", "e": 0.003, "jobs": 2},
        # the benchmark: 1024 trajectories of the 20-qubit noisy QFT
        {"name": "mc_qft_n20_c64_t1024", "kind": "mc", "circuit": "qft", "iterations": 0, "n": 20, "batch": 1024, "dtype": "c64", "e": 0.01, "jobs": 0},
        # a circuit wider than two windows, an odd number of trajectories
        {"name": "mc_qft_n23_c64_t27", "kind": "mc", "circuit": "qft", "iterations": 0, "n": 23, "batch": 27, "dtype": "c64", "e": 0.01, "jobs": 0},
        # the double-precision form that complex64 results are compared with
        {"name": "mc_qft_n18_c128_t75", "kind": "mc", "circuit": "qft", "iterations": 0, "n": 18, "batch": 75, "dtype": "c128", "e": 0.01, "jobs": 0},
        # noisy Grover search, eight iterations: flips and layers of Hadamards on a dense state, four jobs of a launch
        {"name": "serve_grover_n16_c64_t500", "kind": "mc", "circuit": "grover", "iterations": 8, "n": 16, "batch": 500, "dtype": "c64", "e": 0.01, "jobs": 4},
        # relative states of an 11-qubit QFT: 22 qubits, dense from the start
        {"name": "choi_qft_s11_c64_t40", "kind": "choi", "circuit": "qft", "iterations": 0, "n": 22, "batch": 40, "dtype": "c64", "e": 0.01},
        # fixed rank, Grover on 16 qubits at rank 8: two iterations, 80 channels of real factors
        {"name": "rank_grover_n16_r8", "kind": "rank", "circuit": "grover", "iterations": 2, "n": 16, "ranks": "8", "e": 0.01},
        # five fixed-rank jobs of uneven rank in one launch, complex factors, 120 channels
        {"name": "rank_qft_n15_jobs5", "kind": "rank", "circuit": "qft", "iterations": 0, "n": 15, "ranks": "1,2,3,5,8", "e": 0.006},
        # the exact density matrix of the 14-qubit QFT (4 GiB), the reference for the approximations
        {"name": "density_qft_n14_c128", "kind": "density", "circuit": "qft", "iterations": 0, "n": 14, "dtype": "c128", "e": 0.01, "relax": False},
        # the same in single precision on 13 qubits, then relaxation of every qubit
        {"name": "density_relax_n13_c64", "kind": "density", "circuit": "qft", "iterations": 0, "n": 13, "dtype": "c64", "e": 0.01, "relax": True},
        # circuits of large gates: low, scattered and high targets of each block size on 1 GiB of trajectories
        {"name": "blocks_n21_c64_t64", "kind": "blocks", "n": 21, "batch": 64, "dtype": "c64", "e": 0.01, "targets": "0,1,2,3,4;2,9,16,5;20,11,0;19,3,12,7,15"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gates", "mc", "mc", "mc", "choi", "rank", "rank", "density", "density", "blocks"])
    circuit = rng.choice(["qft", "qft", "grover"])
    e = float("%.3g" % math.exp(rng.uniform(math.log(1e-4), math.log(1e-2))))
    if kind == "gates":
        n = rng.randint(6, 15)
        batch = _log_int(rng, 1, min(32, (1 << 17) >> n))
        return {"kind": kind, "circuit": circuit, "iterations": 1 if circuit == "grover" else 0, "n": n, "batch": batch, "dtype": rng.choice(["c64", "c128"]), "e": e}
    if kind == "mc":
        dtype = rng.choice(["c64", "c64", "c64", "c128"])
        n = rng.randint(10, 26 if dtype == "c64" else 21)
        it = rng.randint(1, 8) if circuit == "grover" else 0
        amps = (1 << 30 if dtype == "c64" else 1 << 25) // (1 if it == 0 else 4 * it)
        batch = _log_int(rng, 1, max(1, min(1500, amps >> n)))
        jobs = rng.choice([0, 0, 1, 3])
        return {"kind": kind, "circuit": circuit, "iterations": it, "n": n, "batch": batch, "dtype": dtype, "e": e, "jobs": min(jobs, batch)}
    if kind == "choi":
        n = 2 * rng.randint(5, 11)
        return {"kind": kind, "circuit": "qft", "iterations": 0, "n": n, "batch": _log_int(rng, 1, min(1000, (1 << 27) >> n)), "dtype": "c64", "e": e}
    if kind == "rank":
        n = rng.randint(9, 18)
        most = max(1, min(8, (1 << 20) >> n))
        ranks = [rng.randint(1, 8)]
        while len(ranks) < most and sum(ranks) < (3 << 19) >> n and rng.random() < 0.6:
            ranks.append(rng.randint(1, 8))
        return {"kind": kind, "circuit": circuit, "iterations": 1 if circuit == "grover" else 0, "n": n, "ranks": ",".join(map(str, ranks)), "e": e}
    if kind == "density":
        dtype = rng.choice(["c64", "c128"])
        return {"kind": kind, "circuit": circuit, "iterations": 1 if circuit == "grover" else 0, "n": rng.randint(6, 14 if dtype == "c64" else 13), "dtype": dtype, "e": e, "relax": rng.random() < 0.5}
    dtype = rng.choice(["c64", "c64", "c128"])
    n = rng.randint(10, 24)
    targets = ";".join(",".join(map(str, rng.sample(range(n), rng.randint(3, 5)))) for _ in range(rng.randint(1, 5)))
    batch = _log_int(rng, 1, max(1, min(1000, (1 << 27 if dtype == "c64" else 1 << 23) >> n)))
    return {"kind": "blocks", "n": n, "batch": batch, "dtype": dtype, "e": e, "targets": targets}


# ------------------------------------------------------------------ inputs

def _qubits(case):
    """Qubits the circuit acts on (the system half of a relative state)."""
    return case["n"] // 2 if case["kind"] == "choi" else case["n"]


def _ops(case, marked=1):
    n = _qubits(case)
    return inputs.qft_circuit(n) if case["circuit"] == "qft" else inputs.grover_circuit(n, case["iterations"], marked)


def _draws(case, seed):
    """The seeded inputs of a case: noise key, basis starts, marked items, and per-member values of a mixed launch."""
    rng = np.random.default_rng([seed, 17])
    n = _qubits(case)
    d = {"key": int(rng.integers(1 << 62))}
    jobs = max(1, case.get("jobs", 0)) if case["kind"] != "rank" else len(case["ranks"].split(","))
    grover = case.get("circuit") == "grover"
    d["x0"] = [0 if grover else int(v) for v in rng.integers(1 << n, size=jobs)]
    d["marked"] = [int(v) for v in rng.integers(1, 1 << n, size=jobs)]
    d["keys"] = [int(v) for v in rng.integers(1 << 62, size=jobs)]
    d["es"] = [float(v) for v in case["e"] * rng.uniform(0.3, 1.0, size=jobs)]
    return d


def _members(case, d):
    """Job of each member of a mixed launch, and the member's counter within its job."""
    jobs = case["jobs"]
    job = np.arange(case["batch"]) * jobs // case["batch"]
    return job, np.arange(case["batch"]) - np.searchsorted(job, job)


def _unitaries(case, seed):
    """(targets, U, qubit of the noisy Hadamard after the block) of each block."""
    rng = np.random.default_rng([seed, 23])
    out = []
    for text in case["targets"].split(";"):
        t = [int(v) for v in text.split(",")]
        D = 1 << len(t)
        q, r = np.linalg.qr(rng.normal(size=(D, D)) + 1j * rng.normal(size=(D, D)))
        out.append((t, q * (np.diag(r) / abs(np.diag(r))), int(rng.integers(case["n"]))))
    return out


class State:
    """Handles and plan of one prepared case, released with it."""

    def __init__(self, case):
        self.case, self.h, self.plan, self.refs = case, None, None, []

    def __del__(self):
        if self.plan:
            qs.qs_plan_destroy(self.plan)
        for r in self.refs + ([self.h] if self.h else []):
            qs.qs_destroy(r)


def _set_reference(h, n, ops, x0, dtype):
    ref = circuits.ideal_reference(n, ops, x0, dtype)
    qs.qs_set_reference_from(h, ref)
    qs.qs_synchronize(h)
    qs.qs_destroy(ref)


def prepare(case, seed):
    s = State(case)
    kind, n = case["kind"], case["n"]
    dtype = DTYPES[case.get("dtype", "c128")]
    d = s.draws = _draws(case, seed)
    if kind in ("gates", "mc", "choi", "blocks"):
        s.h = qs.qs_create(n, case["batch"], 0, qs.QS_STATEVEC, dtype)
    if kind == "gates":
        s.ops = _ops(case, d["marked"][0])
    elif kind == "mc":
        jobs = case["jobs"]
        s.plan = qs.qs_plan_create(s.h, circuits.to_gates(_ops(case, d["marked"][0]), per_member_flip=jobs > 0))
        if jobs == 0:
            _set_reference(s.h, n, _ops(case, d["marked"][0]), d["x0"][0], dtype)
        else:
            s.refs = [circuits.ideal_reference(n, _ops(case, d["marked"][j]), d["x0"][j], dtype) for j in range(jobs)]
            job, s.traj = _members(case, d)
            s.e, s.keys = np.array(d["es"])[job], np.array(d["keys"], dtype=np.uint64)[job]
            s.x0, s.marked = np.array(d["x0"], dtype=np.uint64)[job], np.array(d["marked"], dtype=np.uint64)[job]
            s.spans = [(int(np.searchsorted(job, j)), int((job == j).sum())) for j in range(jobs)]
    elif kind == "choi":
        s.plan = qs.qs_plan_create(s.h, circuits.to_gates(_ops(case)))
        ref = qs.qs_create(n, 1, 0, qs.QS_STATEVEC, dtype)
        qs.qs_set_maximally_entangled(ref)
        ideal = qs.qs_plan_create(ref, circuits.to_gates([Op(o.kind, o.qubits, o.theta, o.index, False) for o in _ops(case)]))
        qs.qs_plan_run(ideal, 0.0, 0, 0)
        qs.qs_synchronize(ref)
        qs.qs_plan_destroy(ideal)
        qs.qs_set_reference_from(s.h, ref)
        qs.qs_synchronize(s.h)
        qs.qs_destroy(ref)
    elif kind == "rank":
        ranks = [int(r) for r in case["ranks"].split(",")]
        J = len(ranks)
        s.h = qs.qs_create(n, J, max(ranks), qs.QS_FIXED_RANK, dtype)
        qs.qs_set_member_ranks(s.h, ranks)
        qs.qs_set_member_noise(s.h, d["es"], d["keys"], [0] * J, d["marked"])
        s.plan = qs.qs_plan_create(s.h, circuits.to_gates(_ops(case), per_member_flip=True))
        s.refs = [circuits.ideal_reference(n, _ops(case, d["marked"][j]), d["x0"][j], dtype) for j in range(J)]
    elif kind == "density":
        s.h = qs.qs_create(n, 1, 0, qs.QS_DENSITY, dtype)
        ops = _ops(case, d["marked"][0])
        s.plan = qs.qs_plan_create(s.h, circuits.to_gates(ops))
        _set_reference(s.h, n, ops, d["x0"][0], dtype)
    else:
        s.blocks = _unitaries(case, seed)
        ref = qs.qs_create(n, 1, 0, qs.QS_STATEVEC, dtype)
        qs.qs_set_basis_state(ref, d["x0"][0])
        for t, U, q in s.blocks:
            qs.qs_apply_gate(ref, t, U)
            qs.qs_apply_gate(ref, (q,), circuits.hadamard())
        qs.qs_set_reference_from(s.h, ref)
        qs.qs_synchronize(s.h)
        qs.qs_destroy(ref)
    return s


RELAX = (0.1, 3.0, 2.0)      # t, T1, T2


def run(s):
    case, h, d = s.case, s.h, s.draws
    kind = case["kind"]
    single = case.get("dtype", "c128") == "c64"
    if kind == "gates":
        qs.qs_set_basis_state(h, d["x0"][0])
        circuits.apply_ops(h, s.ops, case["e"], d["key"])
        psi = qs.qs_get_state(h)
        return {"state": psi.astype(np.complex64) if single else psi}
    if kind == "mc" and case["jobs"] == 0:
        qs.qs_set_basis_state(h, d["x0"][0])
        f = qs.qs_plan_run_fidelity(s.plan, case["e"], d["key"], 0, h)
    elif kind == "mc":
        qs.qs_set_member_noise(h, s.e, s.keys, s.traj, s.marked)
        qs.qs_set_basis_states(h, s.x0)
        qs.qs_plan_run(s.plan, 0.0, 0, 0, h)
        f = np.concatenate([qs.qs_fidelity_ref(h, s.refs[j], a, c) for j, (a, c) in enumerate(s.spans)])
    elif kind == "choi":
        qs.qs_set_maximally_entangled(h)
        f = qs.qs_plan_run_fidelity(s.plan, case["e"], d["key"], 0, h)
    elif kind == "rank":
        qs.qs_set_basis_states(h, d["x0"])
        qs.qs_plan_run(s.plan, 0.0, 0, 0, h)
        f = np.concatenate([qs.qs_fidelity_ref(h, s.refs[j], j, 1) for j in range(len(s.refs))])
        return {"fidelity": f, "trace": qs.qs_trace(h)}
    elif kind == "density":
        qs.qs_set_basis_state(h, d["x0"][0])
        qs.qs_plan_run(s.plan, case["e"], 0, 0, h)
        if case["relax"]:
            qs.qs_apply_relaxation(h, list(range(case["n"])), *RELAX)
        f, t = qs.qs_fidelity_stored(h), qs.qs_trace(h)
        return {"fidelity": f.astype(np.float32) if single else f, "trace": t.astype(np.float32) if single else t}
    else:
        qs.qs_set_basis_state(h, d["x0"][0])
        for g, (t, U, q) in enumerate(s.blocks):
            qs.qs_apply_gate(h, t, U)
            qs.qs_apply_noisy_gate(h, (q,), circuits.hadamard(), qs.QS_NOISE_ROTATION, case["e"], d["key"], g)
        f = qs.qs_fidelity_stored(h)
    return {"fidelity": f.astype(np.float32) if single else f}


def work(case):
    """Bytes: the result written once, a given state and the reference read once.  Operations: one complex product per
    amplitude of the result and one for the fidelity at least; a dense circuit's own gates on top."""
    kind, N = case["kind"], 1 << case["n"]
    es = ESIZE[case.get("dtype", "c128")]
    if kind == "rank":
        ranks = [int(r) for r in case["ranks"].split(",")]
        chan = sum(o.noisy for o in _ops(case))
        per = 2 if case["circuit"] == "grover" else 8            # real or complex multiply-add
        flops = sum(chan * N * per * (r * (r + 1) / 2 + r * r) for r in ranks)
        return {"bytes": float(N * 16 * (sum(ranks) + len(ranks))), "flops": float(flops)}
    if kind == "density":
        entries = N * (N + 1) // 2                               # Hermitian
        chan = sum(o.kind == "H" for o in _ops(case))
        return {"bytes": float(N * N * es + N * es), "flops": float(entries * (12 * chan + 8))}
    amps = N * case["batch"]
    out = {"bytes": float(amps * es + N * es), "flops": float(16 * amps)}
    if kind == "gates":
        out["bytes"] = float(amps * es)
    elif kind == "choi" or case.get("circuit") == "grover":
        h = sum(o.kind == "H" for o in _ops(case))
        out["flops"] += amps * 6.0 * h
    elif kind == "blocks":
        out["flops"] += float(amps) * sum(8 * (1 << len(t.split(","))) + 12 for t in case["targets"].split(";"))
    return out


# ------------------------------------------- the same in 64 bits, in plain torch

def _philox(key, traj, gate):
    """xi_a of Philox4x32-10 (Salmon et al., SC'11) and Box-Muller; traj and key: arrays."""
    m32 = np.uint64(0xFFFFFFFF)
    traj, key = np.broadcast_arrays(np.asarray(traj, dtype=np.uint64), np.asarray(key, dtype=np.uint64))
    c = [traj & m32, traj >> np.uint64(32), np.full_like(traj, gate & 0xFFFFFFFF), np.full_like(traj, gate >> 32)]
    k0, k1 = key & m32, key >> np.uint64(32)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m32]
    u = [(((hi << np.uint64(32)) | lo) >> np.uint64(11)).astype(np.float64) for hi, lo in ((c[0], c[1]), (c[2], c[3]))]
    u1, u2 = (u[0] + 0.5) * 2.0 ** -53, (u[1] + 0.5) * 2.0 ** -53
    return np.sqrt(-2.0 * np.log(u1)) * np.cos(2.0 * np.pi * u2)


_DEV = "cuda"
_H = np.array([[1.0, 1.0], [1.0, -1.0]]) / math.sqrt(2.0)


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=_DEV)


def _one(psi, q, M):
    """M (batch or 1, 2, 2) on qubit q of psi (batch, 2^n), in place."""
    v = psi.view(psi.shape[0], -1, 2, 1 << q)
    M = _t(M)[:, :, :, None, None]
    a, b = v[:, :, 0], v[:, :, 1]
    x = M[:, 0, 0] * a + M[:, 0, 1] * b
    v[:, :, 1] = M[:, 1, 0] * a + M[:, 1, 1] * b
    v[:, :, 0] = x


def _both(psi, j, k):
    """View of the amplitudes of psi (batch, 2^n) with qubits j > k set."""
    return psi.view(psi.shape[0], -1, 2, 1 << (j - k - 1), 2, 1 << k)[:, :, 1, :, 1]


def _trajectories(psi, ops, e, key, traj, marked=None):
    """The noisy circuit (e = 0: ideal) on psi (batch, 2^n), in place; e, key, traj (and marked) per member."""
    e = np.asarray(e, dtype=np.float64)
    rows = torch.arange(psi.shape[0], device=_DEV)
    for g, o in enumerate(ops):
        if o.kind == "FLIP":
            at = marked if marked is not None and o.index != 0 else np.full(psi.shape[0], o.index)
            psi[rows, _t(np.asarray(at, dtype=np.int64))] *= -1
            continue
        a = e * _philox(key, traj, g)
        if o.kind == "H":
            c, s = np.cos(a), np.sin(a)
            _one(psi, o.qubits[0], _H @ np.stack([np.stack([c, s], -1), np.stack([-s, c], -1)], -2))
        else:
            _both(psi, *o.qubits).mul_(_t(np.exp(-1j * (o.theta + a)))[:, None, None, None])
    return psi


def _basis(xs, n):
    psi = torch.zeros((len(xs), 1 << n), dtype=torch.complex128, device=_DEV)
    psi[torch.arange(len(xs), device=_DEV), _t(np.asarray(xs, dtype=np.int64))] = 1
    return psi


def _omega(batch, n):
    m = n // 2
    psi = torch.zeros((batch, 1 << n), dtype=torch.complex128, device=_DEV)
    i = torch.arange(1 << m, device=_DEV)
    psi[:, i + (i << m)] = 2.0 ** (-m / 2.0)
    return psi


def _ideal(psi, ops, marked=None):
    return _trajectories(psi, ops, np.zeros(1), 0, 0, marked)[0]


def _overlaps(psi, ref):
    return ((psi @ ref.conj()).abs() ** 2).cpu().numpy()


def _exact_mc(case, seed):
    d, n = _draws(case, seed), case["n"]
    B, kind = case["batch"], case["kind"]
    if case.get("jobs", 0):
        job, traj = _members(case, d)
    else:
        job, traj = np.zeros(B, dtype=int), np.arange(B)
    own = case.get("jobs", 0) > 0
    es = np.array(d["es"])[job] if own else np.full(B, case["e"])
    keys = np.array(d["keys"], dtype=np.uint64)[job] if own else np.full(B, d["key"], dtype=np.uint64)
    x0, marked = np.array(d["x0"])[job], np.array(d["marked"])[job]
    ops = _ops(case, d["marked"][0])
    out = []
    chunk = max(1, (1 << 27) >> n)
    refs = {}
    for a in range(0, B, chunk):
        m = slice(a, min(B, a + chunk))
        psi = _omega(len(es[m]), n) if kind == "choi" else _basis(x0[m], n)
        _trajectories(psi, ops, es[m], keys[m], traj[m], marked[m])
        if kind == "gates":
            out.append(psi.cpu().numpy().reshape(-1))
            continue
        for j in sorted(set(job[m])):
            if j not in refs:
                refs[j] = _ideal(_omega(1, n) if kind == "choi" else _basis([d["x0"][j]], n), ops, [d["marked"][j]])
            out.append(_overlaps(psi[_t(np.nonzero(job[m] == j)[0])] if own else psi, refs[j]))
    return {"state" if kind == "gates" else "fidelity": np.concatenate(out)}


def _channel(o, e):
    """Kraus operators of a noisy gate's average over xi."""
    if o.kind == "H":
        q = math.exp(-2.0 * e * e)
        return [math.sqrt(0.5 * (1 + q)) * _H, math.sqrt(0.5 * (1 - q)) * _H @ np.array([[0.0, 1.0], [-1.0, 0.0]])]
    return math.exp(-e * e)


def _leading(G, keep):
    """Leading eigenvectors of G; eigenvalues within 1e-10 of the largest form a cluster whose basis is Gram-Schmidt of
    the axes projected on it, as qs_truncate_rank defines it."""
    lam, V = np.linalg.eigh(G)
    lam, V = lam[::-1], V[:, ::-1]
    out, i = [], 0
    while len(out) < keep:
        k = i + 1
        while k < len(lam) and lam[i] - lam[k] <= 1e-10 * lam[0]:
            k += 1
        P, got = V[:, i:k] @ V[:, i:k].conj().T, []
        for least in (1e-3, 1e-8):
            for j in range(len(lam)):
                if len(got) < k - i:
                    v = P[:, j] - sum((q * np.vdot(q, P[:, j]) for q in got), np.zeros(len(lam)))
                    if np.linalg.norm(v) > least:
                        got.append(v / np.linalg.norm(v))
        out, i = out + got, k
    return np.stack(out[:keep], axis=1)


def _exact_rank(case, seed):
    d, n = _draws(case, seed), case["n"]
    fid, tr = [], []
    for j, r in enumerate(int(v) for v in case["ranks"].split(",")):
        ops = _ops(case, d["marked"][j])
        L = _basis([d["x0"][j]], n)                               # columns as rows
        for o in ops:
            if o.kind == "FLIP":
                L[:, o.index] *= -1
                continue
            parts = [L.clone(), L]
            if o.kind == "H":
                for p, E in zip(parts, _channel(o, d["es"][j])):
                    _one(p, o.qubits[0], E[None].astype(complex))
            else:
                P, f = _channel(o, d["es"][j]), np.exp(-1j * o.theta)
                _both(parts[0], *o.qubits).mul_(complex(f * math.sqrt(P)))
                kept = _both(parts[1], *o.qubits).clone()
                parts[1].zero_()
                _both(parts[1], *o.qubits).copy_(kept * complex(f * math.sqrt(1 - P)))
            Lp = torch.cat(parts)
            W = _leading((Lp.conj() @ Lp.T).cpu().numpy(), min(r, Lp.shape[0]))
            L = _t(W.T) @ Lp
        ref = _ideal(_basis([d["x0"][j]], n), ops)
        fid.append(float(_overlaps(L, ref).sum()))
        tr.append(float((L.abs() ** 2).sum()))
    return {"fidelity": np.array(fid), "trace": np.array(tr)}


def _exact_density(case, seed):
    d, n, e = _draws(case, seed), case["n"], case["e"]
    N = 1 << n
    ops = _ops(case, d["marked"][0])
    x = d["x0"][0]
    rho = _basis([x * N + x], 2 * n)
    for o in ops:
        if o.kind == "FLIP":
            m = rho.view(N, N)
            m[o.index] *= -1
            m[:, o.index] *= -1
        elif o.kind == "H":
            parts = [rho.clone(), rho]
            for p, E in zip(parts, _channel(o, e)):
                _one(p, o.qubits[0], E[None])
                _one(p, o.qubits[0] + n, E[None])
            rho = parts[0].add_(parts[1])
        else:
            P, f = _channel(o, e), np.exp(-1j * o.theta)
            a, b = o.qubits
            v = rho.view(-1, 2, 1 << (a - b - 1), 2, 1 << b, 1 << (n - 1 - a), 2, 1 << (a - b - 1), 2, 1 << b)
            v[:, 1, :, 1] *= complex(f * math.sqrt(P))
            v[:, :, :, :, :, :, 1, :, 1] *= complex(f.conjugate() * math.sqrt(P))
            v[:, 1, :, 1][:, :, :, :, 1, :, 1] *= 1.0 / P
    if case["relax"]:
        t, T1, T2 = RELAX
        keep, c = math.exp(-t / T1), math.exp(-t / T2)
        for q in range(n):
            v = rho.view(N >> (q + 1), 2, (1 << q) * (N >> (q + 1)), 2, 1 << q)
            v[:, 0, :, 0] += (1.0 - keep) * v[:, 1, :, 1]
            v[:, 1, :, 1] *= keep
            v[:, 0, :, 1] *= c
            v[:, 1, :, 0] *= c
    m = rho.view(N, N)
    ref = _ideal(_basis([x], n), ops)
    return {"fidelity": np.array([float((ref.conj() @ (m @ ref)).real)]), "trace": np.array([float(m.diagonal().sum().real)])}


def _exact_blocks(case, seed):
    d, n, B = _draws(case, seed), case["n"], case["batch"]
    blocks = _unitaries(case, seed)

    def circuit(psi, e, traj):
        for g, (t, U, q) in enumerate(blocks):
            front = [1 + n - 1 - v for v in reversed(t)]
            v = psi.view([psi.shape[0]] + [2] * n).movedim(front, list(range(len(t))))
            psi = (_t(U) @ v.reshape(1 << len(t), -1)).view(v.shape).movedim(list(range(len(t))), front).reshape(psi.shape[0], -1)
            a = e * _philox(d["key"], traj, g)
            c, s = np.cos(a), np.sin(a)
            _one(psi, q, _H @ np.stack([np.stack([c, s], -1), np.stack([-s, c], -1)], -2))
        return psi

    ref = circuit(_basis([d["x0"][0]], n), 0.0, np.zeros(1))[0]
    out = []
    chunk = max(1, (1 << 27) >> n)
    for a in range(0, B, chunk):
        traj = np.arange(a, min(B, a + chunk))
        out.append(_overlaps(circuit(_basis([d["x0"][0]] * len(traj), n), case["e"], traj), ref))
    return {"fidelity": np.concatenate(out)}


def exact(case, seed):
    with torch.no_grad():
        return {"rank": _exact_rank, "density": _exact_density, "blocks": _exact_blocks}.get(case["kind"], _exact_mc)(case, seed)
