"""A cache file of a build with other launch rules: its choice is not taken over."""
import hashlib
import json
from types import SimpleNamespace

import torch

from paper_1611_09704_gb300 import autotune


def test_a_choice_made_under_other_rules_is_tuned_again(tmp_path, monkeypatch):
    path = str(tmp_path / "t.json")
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d=None: "fake")
    specs = [SimpleNamespace(x=torch.empty((2, 50)), widths=[1, 2], threshold=6.0, sigma_mode=0,
                             scope=0, nmax=0)]
    # the key as it was before there were versions: device and batch alone
    desc = [["torch.float32", 2, 50, [1, 2], 6.0, 0, 0, 0]]
    old = hashlib.sha1(json.dumps(["fake", desc], sort_keys=True).encode()).hexdigest()
    slow = {"ctas_per_sm": 0, "group_scale": 1, "tile_threads": 128}
    autotune.save_cache(path, {old: {"tuning": slow, "timings_ms": {}},
                               "another batch": {"tuning": slow, "timings_ms": {}}})
    # the device of a CPU tensor is named by its type
    monkeypatch.setattr(autotune, "batch_key", lambda s, name, key=autotune.batch_key: key(s, "fake"))
    r = autotune.autotune(specs, 10, cache_path=path,
                          timer=lambda s, c, t, n: 1.0 + (t["tile_threads"] == 128))
    assert not r["cached"] and r["tuning"]["tile_threads"] == 256
    assert autotune.load_cache(path)["another batch"]["tuning"] == slow
    assert autotune.autotune(specs, 10, cache_path=path)["cached"]
