"""Shapes stored for other propagation kernels are not applied (host logic)."""
import json

from paper_2507_04115_gb300 import tunecache


def test_keys_of_other_kernels_do_not_match(tmp_path):
    key = tunecache.batch_key([(4096, 0.15, 1.19, 1.0, 100)], 0, 0, 0, "GB300")
    fields = json.loads(key)
    del fields["sweeps"]
    old = json.dumps(fields, sort_keys=True, separators=(",", ":"))   # the key before the generation was part of it
    path = str(tmp_path / "tune.json")
    with open(path, "w") as fh:
        json.dump({"version": 1, "shapes": {old: {"warps_per_cta": 8, "ctas_per_sm": 1, "slice_steps": 16}}}, fh)
    cache = tunecache.TuneCache(path)
    assert cache.get(old) is not None and cache.get(key) is None
