"""The autotuner where the tiled form runs no tiles: nothing to choose, nothing to log, nothing to
learn from (host logic only)."""
import importlib.util
import os

import paper_1004_5059_gb300 as tv
from paper_1004_5059_gb300 import autotune

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class FakeSim:
    nx, ny, velset, storage = 64, 64, tv.TVLBM_D2Q16, tv.TVLBM_FP32

    def __init__(self, tiles):
        self.tiles, self.selected = tiles, 2

    def runs_tiles(self):
        return self.tiles

    def tile(self):
        return self.selected

    def set_tile(self, config):
        self.selected = config


def test_no_trials_without_tiles(monkeypatch, tmp_path):
    log = str(tmp_path / "log.jsonl")
    timed = []
    monkeypatch.setattr(autotune, "time_config", lambda sim, cfg, steps, repeats: timed.append(cfg) or (4 - cfg) * 1e-6)
    monkeypatch.setattr(autotune, "tile_shapes", lambda sim: [(32, 8, 4), (32, 16, 4), (64, 8, 2), (64, 16, 4)])
    sim = FakeSim(False)
    r = autotune.autotune(sim, log_path=log, form="tiled")
    assert timed == [2] and r["best"] == sim.selected == 2 and not os.path.exists(log)
    assert r["trials"] == [{"config": 2, "tile": None, "s_per_step": 2e-6}]
    sim = FakeSim(True)
    r = autotune.autotune(sim, log_path=log, form="tiled")
    assert r["best"] == sim.selected == 3 and len(autotune.read_log(log)) == 4


def test_predict_leaves_out_grids_without_tiles():
    def rec(n, cfg, t, form="tiled"):
        return {"nx": n, "ny": n, "velset": tv.TVLBM_D2Q16, "storage": tv.TVLBM_FP32, "form": form, "config": cfg,
                "tile": [32, 8, 4], "s_per_step": t}
    # 512 x 512 runs without tiles: its winner is noise and must not reach 1024 x 1024
    records = [rec(512, 3, 1e-6), rec(4096, 1, 1e-6)]
    p = autotune.predict(records, 1024, 1024, tv.TVLBM_D2Q16, tv.TVLBM_FP32, "tiled")
    assert p["config"] == 1 and p["from"] == [4096, 4096]
    assert autotune.predict(records[:1], 1024, 1024, tv.TVLBM_D2Q16, tv.TVLBM_FP32, "tiled") is None
    flow = [rec(512, 3, 1e-6, "flow")]  # the dataflow form runs tiles on every size
    assert autotune.predict(flow, 1024, 1024, tv.TVLBM_D2Q16, tv.TVLBM_FP32, "flow")["config"] == 3


def test_bench_says_where_no_tiles_ran():
    spec = importlib.util.spec_from_file_location("bench_for_labels", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    assert bench.form_label(FakeSim(False), "tiled") == "tiled (without tiles)"
    assert bench.form_label(FakeSim(True), "tiled") == "tiled" and bench.form_label(FakeSim(False), "strip") == "strip"
    assert bench.form_tile(tv, FakeSim(False), "tiled", 0) is None
    assert bench.form_tile(tv, FakeSim(False), "strip", 0) == [128, 1, 1]
