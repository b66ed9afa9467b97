"""The benchmark line says what ran: the region-merging engine has no schedule, and
no wavefront setting or cost model touches its step."""
import os
import sys
from types import SimpleNamespace

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

SETTINGS = {"block_h": 128, "bands": 4, "scan_pairs": 1, "grid": 608}
META = {"tiles": 20000, "variants": [1, 2], "epochs": 200}


def work(fetch):
    return {"phase_ns": {"load": 5, "scan": 1, "seed": 1, "queue": 1, "write": 1, "fetch": fetch}}


def test_the_engine_is_read_off_the_counters():
    assert bench.ran_merging([work(0), work(0)])
    assert not bench.ran_merging([work(0), work(7)])


def test_a_merging_step_names_no_schedule():
    c = bench.schedule_config(True, SETTINGS, "learned", META, None)
    assert c["engine"] == "region merging"
    for key in ("schedule", "cost_model", *SETTINGS):
        assert key in c and c[key] is None, key
    assert c["autotuned"] is False


@pytest.mark.parametrize("schedule,meta,tuned", [("learned", META, None), ("plain", None, (64, 4, 1, 0))])
def test_a_wavefront_step_names_its_schedule(schedule, meta, tuned):
    c = bench.schedule_config(False, SETTINGS, schedule, meta, tuned)
    assert c["engine"] == "wavefront" and c["schedule"] == schedule and c["autotuned"] == (tuned is not None)
    assert all(c[k] == v for k, v in SETTINGS.items())
    assert c["cost_model"] == ({"tiles": 20000, "variants": [1, 2]} if meta else None)


def test_launches_of_a_merging_batch():
    def tiles(*sizes, conn=8):
        return [SimpleNamespace(H=h, W=w, conn=conn) for h, w in sizes]
    assert bench.merging_launches(tiles((64, 64), (3, 60))) == 1             # single blocks only
    assert bench.merging_launches(tiles((64, 64), (65, 64))) == 3
    assert bench.merging_launches(tiles((65, 64)) + tiles((64, 64), conn=4)) == 4
    assert bench.merging_launches(tiles(*[(4096, 4096)] * 16)) == 3           # 65536 blocks
    assert bench.merging_launches(tiles(*[(4096, 4096)] * 17)) == 6
