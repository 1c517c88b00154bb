"""The benchmark's look-up in the recorded DRAM traffic (CPU)."""

import json

import pytest

import bench
from paper_2009_09500_gb300 import build, vox


@pytest.fixture
def record(tmp_path, monkeypatch):
    build.build_library()
    vox.load()
    (tmp_path / "profiles").mkdir()
    tuning = {"run_len": 32, "volume_path": 0, "ctas_per_sm": 0, "list_runs": 0}
    ent = {"source_hash": "h", "tuning": tuning, "dram_bytes_per_launch": 5.0}
    atomic = {**ent, "tuning": {**tuning, "volume_path": vox.VOLUME_ATOMIC}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps({"w/a": ent, "w/b": ent, "w/c": atomic}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "_kernel_source_hash", lambda: "h")
    yield
    vox.vox_reset_tuning()


@pytest.mark.parametrize("tuning,found", [((0, 0, 0, 0), True), ((32, 0, 0, 0), True), ((64, 0, 0, 1), True),
                                          ((32, 0, 4, 2), True),
                                          ((32, 0, 2, 0), False), ((32, 1, 0, 0), False)])
def test_record_is_found_under_equal_launches(record, tuning, found):
    vox.vox_set_tuning(*tuning)
    assert bench._recorded_field("w", ["a", "b"], "dram_bytes_per_launch") == (10.0 if found else None)


@pytest.mark.parametrize("run_len,found", [(32, True), (64, False)])
def test_atomics_keep_their_run_length(record, run_len, found):
    vox.vox_set_tuning(run_len, vox.VOLUME_ATOMIC, 0, 0)
    assert bench._recorded_field("w", ["c"], "dram_bytes_per_launch") == (5.0 if found else None)
    assert bench._recorded_field("w", ["a"], "dram_bytes_per_launch") is None
