"""The traffic bench.py reports belongs to the launch it times."""
import json

import bench


def test_traffic_of_the_timed_launch(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    summary = {"launch": "32,4,11,2", "dram_bytes_per_launch_full_size": 123.0,
               "kernel_source_hash": bench.kernel_source_hash()}
    (tmp_path / "profiles" / "k.json").write_text(json.dumps(summary))
    (tmp_path / "profiles" / "old.json").write_text(json.dumps(dict(summary, kernel_source_hash="0" * 16)))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda h=bench.kernel_source_hash(): h)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    same = {"bx": 32, "by": 4, "variant": 11, "tiles": 2, "ms_per_step": 0.1}
    other = dict(same, bx=64)
    assert bench.traffic_fields("k", same) == {"traffic": 123.0}
    assert bench.traffic_fields("k", other) == {"traffic": None, "traffic_of_other_launch":
                                                {"bytes": 123.0, "launch": "32,4,11,2"}}
    assert bench.profiled_traffic("k", other) is None and bench.profiled_traffic("k") == 123.0
    for name in ("old", "none"):
        assert bench.traffic_fields(name, same) == {"traffic": None}
