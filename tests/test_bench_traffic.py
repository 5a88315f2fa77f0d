"""The benchmark combines a captured DRAM traffic with a measured launch time only while
the capture describes the kernel that runs: any change of a kernel header, or launches
that advance by another number of steps, set it aside (CPU only)."""
import json
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
CSRC = os.path.join("paper_2307_11752_gb300", "csrc")
HEADERS = sorted(f for f in os.listdir(os.path.join(ROOT, CSRC)) if f.endswith((".cuh", ".h")))


@pytest.fixture
def bench(tmp_path, monkeypatch):
    import bench as b

    shutil.copytree(os.path.join(ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(b, "ROOT", str(tmp_path))
    record = tmp_path / "traffic.json"
    monkeypatch.setattr(b, "PROFILE_TRAFFIC", str(record))
    record.write_text(json.dumps({
        "one": {"source_sha": b.kernel_source_sha(), "dram_bytes_per_fluid_cell": 135.0},
        "two": {"source_sha": b.kernel_source_sha(), "dram_bytes_per_fluid_cell": 150.0, "steps_per_launch": 2}}))
    return b


def test_traffic_of_the_captured_kernel_is_used(bench):
    assert bench.profiled_traffic("one", 10, 1.0) == 1350.0
    assert bench.profiled_traffic("two", 10, 2.0) == 1500.0
    assert bench.profiled_traffic("three", 10, 1.0) is None


def test_other_steps_per_launch_set_the_capture_aside(bench):
    assert bench.profiled_traffic("one", 10, 2.0) is None
    assert bench.profiled_traffic("two", 10, 1.0) is None


@pytest.mark.parametrize("name", HEADERS)
def test_any_header_sets_the_capture_aside(bench, tmp_path, name):
    with open(tmp_path / CSRC / name, "a") as fh:
        fh.write("// edited\n")
    assert bench.profiled_traffic("one", 10, 1.0) is None
