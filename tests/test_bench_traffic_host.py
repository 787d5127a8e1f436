"""The benchmark finds the committed ncu figures of the split-axis classes, which run in both sweeps with one class number."""
import importlib.util
import json
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_traffic", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


@pytest.mark.parametrize("cls", [8, 9, 10])
def test_split_axis_classes_by_sweep(bench, cls):
    h = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))["kernel_source_hash"]
    got = {}
    for phase in ("forward", "adjoint"):
        got[phase] = [bench.stored_traffic(cls, h, k, phase) for k in ("dram_bytes_per_launch_full", "warp_instructions_per_launch")]
        assert all(v and v > 0 for v in got[phase]), (cls, phase)
        assert bench.stored_traffic(cls, "0" * 16, phase=phase) is None
    assert got["forward"] != got["adjoint"]
    assert bench.stored_traffic(6, h, phase="adjoint") == bench.stored_traffic(6, h)   # one sweep only
