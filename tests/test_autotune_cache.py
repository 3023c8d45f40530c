"""The tuner's cache across versions of the kernels, and timings that scatter (no
GPU: the fakes of test_autotune)."""
import json

from paper_2311_15242_gb300 import autotune as AT
from test_autotune import FakeBatch, FakeSolver, costs, fake_timer


def test_entries_of_other_kernels_are_timed_again(tmp_path):
    path = tmp_path / "tiles.json"
    old = {"d2q9/f32/w128": {"tx": 256, "ty": 1, "sor": 7, "ms_per_step": 1.0},
           "d3q19/bf16/w256/single": {"sor": 2, "ms_per_step": 1.0, "kernels": AT.KERNELS - 1},
           "d2q9/f16/w64": "not an entry"}
    path.write_text(json.dumps(old))
    r = AT.tune(FakeBatch(), [128], timer=fake_timer(costs((64, 4), 2)), cache_path=str(path))
    assert r["source"] == "timed" and (r["tx"], r["ty"], r["sor"]) == (64, 4, 2)
    s = FakeSolver()
    s.storage = "bf16"
    r = AT.tune_single(s, 256, lattice="d3q19", timer=lambda b: 1.0 + b.calls[-1],
                       cache_path=str(path))
    assert r["source"] == "timed" and r["sor"] == 0
    saved = json.loads(path.read_text())
    assert saved["d2q9/f32/w128"]["kernels"] == saved["d3q19/bf16/w256/single"]["kernels"] == AT.KERNELS
    # and used from then on
    def no_timing(_):
        raise AssertionError("timed on a cache hit")
    assert AT.tune(FakeBatch(), [128], timer=no_timing, cache_path=str(path))["source"] == "cache"
    assert AT.tune_single(s, 256, lattice="d3q19", timer=no_timing,
                          cache_path=str(path))["source"] == "cache"


def test_scatter_does_not_choose_a_cell_tile(tmp_path):
    """Tiles that no launch depends on: the timings differ by their scatter only."""
    scatter = iter([1.000, 0.995, 1.008, 0.991, 1.002, 0.997, 1.004, 0.993] + [2.0] * 20)
    r = AT.tune(FakeBatch(), [128], timer=lambda b: next(scatter),
                cache_path=str(tmp_path / "tiles.json"))
    assert (r["tx"], r["ty"], r["sor"]) == (*AT.CELL_TILES[0], 0)


def test_a_run_that_settles_does_not_choose_a_cell_tile(tmp_path):
    """The first steps of a run take more solver rounds, whatever the tile."""
    n = [0]

    def settling(b):
        n[0] += 1
        return 1.0 + 0.5 / n[0]
    r = AT.tune(FakeBatch(), [128], timer=settling, cache_path=str(tmp_path / "tiles.json"))
    assert (r["tx"], r["ty"]) == AT.CELL_TILES[0]
