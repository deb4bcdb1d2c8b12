"""A configuration timed with other kernels is not taken from the cache (host
logic, no GPU)."""

from __future__ import annotations

import json

from paper_2301_10838_gb300 import autotune


def test_entries_of_other_kernels_are_misses(tmp_path, monkeypatch):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("MT_AUTOTUNE_CACHE", str(path))
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda d: "GPU-A")
    old = {"GPU-A|a": {"cfg": 8, "ms": {"0": 2.0}}, "GPU-A|b": {"cfg": 1, "ms": [1.0], "kernels": autotune.KERNELS - 1}}
    path.write_text(json.dumps(old))
    assert autotune.lookup(0, "a") is None and autotune.lookup(0, "b") is None
    autotune.store(0, "a", 0, {"0": 1.0})
    assert autotune.lookup(0, "a") == {"cfg": 0, "ms": {"0": 1.0}}
    assert autotune.lookup(0, "b") is None
    monkeypatch.setattr(autotune, "KERNELS", autotune.KERNELS + 1)
    assert autotune.lookup(0, "a") is None
