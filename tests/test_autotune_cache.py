"""Cached winners of another sweep are not applied."""
import json

import torch


def test_winners_of_another_sweep_are_timed_again(tmp_path, monkeypatch):
    from paper_2103_04856_gb300 import autotune
    dev = torch.cuda.get_device_name() if torch.cuda.is_available() else "cpu"
    cache = tmp_path / "cache.json"
    # as the one-voxel sweep's tuner wrote it: its 13-row tiles
    cache.write_text(json.dumps({f"{dev}|fp32|64x64x64": {"tile_y": 13, "max_run": 0, "sweep_ms": 0.1}}))
    monkeypatch.setattr(autotune, "time_candidate", lambda shapes, cand, **kw: 1.0 if cand["tile_y"] != 16 else 0.5)
    assert autotune.tune([(64, 64, 64)], cache=str(cache))["tile_y"] == 16
    key = autotune.cache_key([(64, 64, 64)])
    monkeypatch.setattr(autotune, "SWEEP", "another")
    assert autotune.cache_key([(64, 64, 64)]) != key
