"""Which cached launch shapes the tuner takes: those timed on this solver, for
this workload. (A stand-in scene; the times are made up.)"""
import types

import pytest

from paper_2011_00459_gb300 import autotune as A


class Bed:
    n, sizes, solver, impact = 1000000, [1000000], (50, 0.0, 10), False

    def __init__(self):
        self.cfg = dict(pgs_blocks=152, pgs_sync=1, colour_blocks=608, pgs_threads=512, pgs_per_thread=2)

    def launch_config(self):
        return dict(self.cfg, max_pgs_blocks=152, max_colour_blocks=1216)

    def set_launch_config(self, **kw):
        self.cfg.update(kw)

    def set_solver(self, *a):
        pass


@pytest.fixture
def sim(monkeypatch):
    import torch

    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(name="NVIDIA GB300", multi_processor_count=152))
    sim = types.SimpleNamespace(g=Bed(), advance=lambda: None)
    monkeypatch.setattr(A, "time_steps", lambda s, steps: 1.0 if s.g.cfg["pgs_threads"] == 512 else 2.0)
    return sim


OLD = {"shape": {"pgs_blocks": 304, "pgs_sync": 1, "colour_blocks": 608, "pgs_threads": 416, "pgs_per_thread": 1}, "ms": 12.1}


def test_an_entry_of_another_solver_is_not_taken(sim, tmp_path, monkeypatch):
    path = str(tmp_path / "tune.json")
    A.store_cache("NVIDIA GB300|n=1000000|scenes=1", OLD, path)  # the key as it was before it named the schedule
    monkeypatch.setattr(A, "SCHEDULE", A.SCHEDULE - 1)
    A.store_cache(A.shape_key("NVIDIA GB300", 1000000, 1), OLD, path)
    monkeypatch.setattr(A, "SCHEDULE", A.SCHEDULE + 1)
    r = A.tune(sim, steps=1, path=path)
    assert r["source"] == "timed" and r["shape"]["pgs_threads"] == 512
    again = A.tune(sim, steps=1, path=path)
    assert again["source"] == "cache" and again["shape"] == r["shape"]


def test_other_shapes_are_another_schedule(sim, tmp_path, monkeypatch):
    path = str(tmp_path / "tune.json")
    A.tune(sim, steps=1, path=path)
    monkeypatch.setattr(A, "SHAPES", A.SHAPES[:-1])
    assert A.tune(sim, steps=1, path=path)["source"] == "timed"


def test_scenes_with_and_without_an_impact_stage(sim, tmp_path):
    path = str(tmp_path / "tune.json")
    A.tune(sim, steps=1, path=path)
    sim.g.impact = True
    assert A.tune(sim, steps=1, path=path)["source"] == "timed"
    assert A.tune(sim, steps=1, path=path)["source"] == "cache"
    sim.g.impact = False
    assert A.tune(sim, steps=1, path=path)["source"] == "cache"
