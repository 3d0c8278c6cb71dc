"""The recorded DRAM traffic of the sweep: counted by passes over memory, and dropped
when a source that the batch kernels are built from or planned by has changed."""
import json
import os

import bench


def _record(tmp_path, monkeypatch):
    path = tmp_path / "traffic.json"
    path.write_text(json.dumps({"passes": {
        "source_hash": bench.kernel_source_hash(),
        "storage": {"f32": {"steps_per_pass": 3, "dram_bytes_per_pass": 1000},
                    "f16d": {"steps_per_pass": 2, "dram_bytes_per_pass": 600}}}}))
    monkeypatch.setattr(bench, "PROFILE_TRAFFIC", str(path))


def test_traffic_counts_passes(tmp_path, monkeypatch):
    _record(tmp_path, monkeypatch)
    assert bench.recorded_traffic("f32", "nearest", 3, 3) == 1000
    assert bench.recorded_traffic("f32", "nearest", 20, 3) == 7000
    assert bench.recorded_traffic("f16d", "nearest", 20, 2) == 6000
    assert bench.recorded_traffic("f32", "nearest", 20, 1) is None  # another pass length
    assert bench.recorded_traffic("bf16d", "nearest", 20, 2) is None
    assert bench.recorded_traffic("f32", "stochastic", 20, 3) is None


def test_traffic_is_dropped_when_the_walk_changes(tmp_path, monkeypatch):
    names = {os.path.basename(p) for p in bench.KERNEL_SOURCES + bench.WALK_SOURCES}
    assert {"lbm_fused.cuh", "lbm_batch.cu", "lbm_batch_kernels.cuh"} <= names
    _record(tmp_path, monkeypatch)
    changed = tmp_path / "lbm_fused.cuh"
    changed.write_text(open(bench.WALK_SOURCES[0]).read() + "\n// changed\n")
    monkeypatch.setattr(bench, "WALK_SOURCES", [str(changed)] + bench.WALK_SOURCES[1:])
    assert bench.recorded_traffic("f32", "nearest", 20, 3) is None
