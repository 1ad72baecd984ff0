"""The autotuner's choice among schedules and the library's own, with a fake device
clock: it never names a schedule that an untouched context beats, and it takes no
timing of other kernels from its cache.
"""
import json

import numpy as np
import pytest

import workloads as W


@pytest.fixture
def tuner(monkeypatch, tmp_path):
    from paper_2411_10751_gb300 import autotune
    clock = [0.0]
    cost = {}

    class Event:
        def __init__(self, **kw):
            self.t = None

        def record(self, stream=None):
            self.t = clock[0]

        def synchronize(self):
            pass

        def elapsed_time(self, other):
            return other.t - self.t

    class Context:
        def __init__(self, *a, **kw):
            self.sched = (0, 0, 0)

        def set_tile(self, *s):
            self.sched = s

        def step(self, n):
            clock[0] += n * cost.get(self.sched, 9.0)

        def set_force_field(self, *a):
            pass

        init = set_force_field
        synchronize = close = cuda_stream = lambda self: None

    monkeypatch.setattr(autotune, "HLBM", Context)
    monkeypatch.setattr(autotune, "CACHE", tmp_path / "autotune.json")
    monkeypatch.setattr(autotune.torch.cuda, "Event", Event)
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda *a: "GPU")

    def run(lattice="D2Q37", nz=1):
        z = np.zeros(1)
        return tuple(autotune.tune(lattice, 64, 64, nz, 0.8, W.source_params(), z, z, z))
    run.cost, run.cache = cost, autotune.CACHE
    return run


@pytest.mark.parametrize("lattice,nz", [("D2Q37", 1), ("D3Q39", 64)])
def test_the_librarys_own_choice_wins_where_it_is_faster(tuner, lattice, nz):
    tuner.cost.update({(0, 0, 0): 2.7, (8, 2, 1): 4.3, (8, 2, 2): 4.6})
    assert tuner(lattice, nz) == (0, 0, 0)
    assert tuner(lattice, nz) == (0, 0, 0)    # and from the cache


def test_a_schedule_is_named_where_it_is_as_fast(tuner):
    tuner.cost.update({(0, 0, 0): 5.00, (8, 2, 2): 5.02, (8, 2, 1): 6.0})
    assert tuner() == (8, 2, 2)


def test_timings_of_other_kernels_are_not_taken(tuner, monkeypatch):
    from paper_2411_10751_gb300 import autotune
    tuner.cost.update({(0, 0, 0): 2.7, (8, 2, 1): 4.3})
    old = {"schedule": [16, 1, 1], "ms_per_step": {}}
    tuner.cache.write_text(json.dumps({"GPU|D2Q37|local|f32|64x64x1": old}))
    assert tuner() == (0, 0, 0)
    tuner.cost[(8, 2, 1)] = 1.0
    assert tuner() == (0, 0, 0)               # the same sources: from the cache
    monkeypatch.setattr(autotune, "_sources", lambda: "other")
    assert tuner() == (8, 2, 1)
