"""The tile autotuner can return the library's defaults (no GPU): a solver
stand-in whose defaults are the fastest tiles keeps them, and a choice cached
when the defaults were not among the candidates is made again."""
import json

import pytest

from paper_2103_08246_gb300 import autotune, binding, inputs

DEFAULTS = {"rhs_planes": 0, "rhs_stages": 8, "afx_planes": 64}


class FakeSolver:
    def __init__(self, wl, precision, tiles=None):
        self.tiles = dict(tiles)

    def step(self, n=1, dt=None):
        pass

    def time_stage(self, stage, nrep=10):
        names = [k for k, v in autotune.STAGE_OF.items() if v == stage]
        return 1.0 + sum(self.tiles[k] != DEFAULTS[k] for k in names)

    def close(self):
        pass


@pytest.mark.parametrize("cached", [False, True])
def test_defaults_that_are_fastest_are_kept(tmp_path, monkeypatch, cached):
    monkeypatch.setattr(binding, "Solver", FakeSolver)
    monkeypatch.setattr(autotune, "_gpu_name", lambda: "test-gpu")
    wl = inputs.small(16, 8, 8)
    cache = tmp_path / "tiles.json"
    if cached:
        old = {"rhs_planes": 16, "rhs_stages": 6, "afx_planes": 64}
        timings = {f"rhs_planes={v}": 1.0 for v in (8, 16, 32, 64)}
        key = f"{wl.nx}x{wl.ny}x{wl.nz}:p{binding.IBM_FP32}:test-gpu"
        cache.write_text(json.dumps({key: {"tiles": old, "timings_ms": timings}}))
    assert autotune.tune(wl, binding.IBM_FP32, cache_path=str(cache), reps=1) == DEFAULTS
