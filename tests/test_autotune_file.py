"""Saved tunings: an entry timed with other kernels is not applied."""
import json

import pytest


@pytest.mark.parametrize("stamp,applied", [(None, 0), ("older", 0), ("same", 1)])
def test_entries_of_other_kernels_are_left_out(tmp_path, monkeypatch, stamp, applied):
    from paper_1306_2461_gb300 import autotune, of
    monkeypatch.setattr(autotune, "_device", lambda: "gpu")
    plan = of.Plan.make(64, 64, 3, 9, 5, bits=12, storage="f16")
    method = autotune._method(plan)
    ent = {"method": method, "size_class": 20, "batch": 8, "candidates": [],
           "best": {"generic_sums": 1, "stage_i2": 0, "blocks_per_sm": 0, "phased": 1, "prefetch": 0, "tile_h": 24,
                    "branches": 1, "fusion": 1, "strip": 1, "ms": 6.9}}
    if stamp:
        ent["kernels"] = autotune.KERNELS - (stamp == "older")
    path = tmp_path / "tune.json"
    path.write_text(json.dumps({"gpu": {autotune._key(method, 20): ent}}))
    of.tuning_clear()
    assert autotune.load(str(path)) == applied
    assert (of.tuning_get(plan, 20) is not None) == bool(applied)
    of.tuning_clear()
