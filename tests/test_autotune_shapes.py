"""Saved autotuner entries and the launch shapes that they were timed against
(GPU): a new market takes an entry of this library's shapes; one without the
field, from before the default shape changed, stays in the cache and in the
saved file but is not taken. No market is timed here."""

import json

import pytest

from synth import make_market

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes,taken", [(None, False), (1, False), (2, True), (3, False)])
def test_entries_apply_to_their_shapes(gpu_lib, tmp_path, shapes, taken):
    import torch
    tu = gpu_lib
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    entry = dict(n_bucket=46, m_bucket=45, kp=64, dtype=0, sms=sms, small_tiles=0, split=3, ms=1.0, ms_default=2.0)
    if shapes is not None:
        entry["shapes"] = shapes
    path = tmp_path / "tuned.json"
    path.write_text('{"tu_autotune": 1, "entries": [\n' + json.dumps(entry) + "\n]}\n")
    tu.tu_autotune_cache_clear()
    try:
        tu.tu_autotune_cache_load(str(path))
        mk = make_market(3000, 2500, 24, sigma=0.5, seed=1, dtype="bf16")  # buckets floor(4 log2): 46, 45
        mkt = tu.from_synth(mk)
        try:
            assert tu.tu_market_get_shape(mkt.handle) == ((0, 3) if taken else (1, 1))
        finally:
            mkt.close()
        tu.tu_autotune_cache_save(str(path))
        saved = json.loads(path.read_text())["entries"]
        assert len(saved) == 1 and saved[0]["shapes"] == (shapes or 1) and saved[0]["split"] == 3
    finally:
        tu.tu_autotune_cache_clear()
