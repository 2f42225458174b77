"""The autotuner's cache, without a GPU: an entry is taken only by the library
version whose paths it was timed on; an entry of another version, or one
without any, is timed again."""
import json

import torch

from paper_2103_17238_gb300 import autotune, sdm

SHAPE = dict(smem_max_sd=4096, warp_cell_max=512, warps_per_block=2)


def _tune(monkeypatch, path, timed):
    tunings = []
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "a GPU")
    monkeypatch.setattr(autotune, "signature", lambda runs: "g15:64")
    monkeypatch.setattr(sdm, "sdm_set_tuning", lambda t: tunings.append(t))
    monkeypatch.setattr(autotune, "time_candidate", lambda runs, steps: timed.append(1) or float(tunings[-1]["mid_max_sd"] + 1))
    rep = autotune.tune([], cache_path=str(path), candidates=[dict(SHAPE, mid_max_sd=16384), dict(SHAPE, mid_max_sd=0)])
    return rep, tunings[-1]


def test_entry_of_this_version(monkeypatch, tmp_path):
    timed = []
    rep, _ = _tune(monkeypatch, tmp_path / "c.json", timed)
    assert not rep["cached"] and len(timed) == 2
    rep, last = _tune(monkeypatch, tmp_path / "c.json", timed)
    assert rep["cached"] and len(timed) == 2 and last["mid_max_sd"] == 0


def test_entries_of_other_versions(monkeypatch, tmp_path):
    path = tmp_path / "c.json"
    timed = []
    old = {"best": dict(SHAPE, mid_max_sd=65536), "ms_per_step": 1.0, "all": []}
    path.write_text(json.dumps({"a GPU|g15:64": old}))
    rep, last = _tune(monkeypatch, path, timed)
    assert not rep["cached"] and len(timed) == 2 and last["mid_max_sd"] == 0
    monkeypatch.setattr(autotune, "PATHS_VERSION", autotune.PATHS_VERSION + 1)
    rep, _ = _tune(monkeypatch, path, timed)
    assert not rep["cached"] and len(timed) == 4
