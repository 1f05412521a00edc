"""What the bench's roofline row is credited with: the pass with the most time, the
kernel that runs in it, and the traffic recorded for it."""
import json

import bench

QFT20 = ["precompute", "pass_high", "precompute", "pass_low"]


def test_bytes_only_where_the_pass_creates_the_whole_state():
    ms = {"precompute": [0.05, 0.0], "pass_high": [0.04], "pass_low": [1.3]}
    kind, kernel, writes = bench.dominant_pass(QFT20, ms, True)
    assert (kind, writes) == ("pass_low", 1) and kernel.startswith("k_outer")
    # no outer product: the pass reads what the first one wrote
    assert bench.dominant_pass(QFT20, ms, False) == ("pass_low", "k_pass_low", None)
    # a pass on part of the support, or several of its kind
    assert bench.dominant_pass(QFT20, {**ms, "pass_high": [2.0]}, True) == ("pass_high", "k_pass_high", None)
    grover = ["precompute", "pass_low"] * 3
    assert bench.dominant_pass(grover, {"precompute": [0.1] * 3, "pass_low": [1.0] * 3}, False) == ("pass_low", "k_pass_low", None)
    # a circuit of one pass
    assert bench.dominant_pass(["precompute", "pass_low"], {"precompute": [0.1], "pass_low": [1.0]}, False) == ("pass_low", "k_pass_low", 1)


def test_traffic_is_of_the_profiled_sources_and_workload(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_1412_2293_gb300" / "csrc"
    csrc.mkdir(parents=True)
    names = ["pass.cuh", "pass_start.cu", "plan.cu", "philox.cuh"]      # k_outer is in plan.cu
    for f in names:
        (csrc / f).write_text(f)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    record = {"source_hash": bench.plan_source_hash(), "workload": "w", "window": 10, "kernels": {"pass_low": 7}}
    (tmp_path / "profiles" / "traffic.txt").write_text(json.dumps(record))
    assert bench.ncu_traffic("pass_low", "w", 10) == 7.0
    assert bench.ncu_traffic("pass_high", "w", 10) is None
    assert bench.ncu_traffic("pass_low", "v", 10) is None and bench.ncu_traffic("pass_low", "w", 11) is None
    for f in names:
        (csrc / f).write_text(f + " changed")
        assert bench.ncu_traffic("pass_low", "w", 10) is None, f
        (csrc / f).write_text(f)
