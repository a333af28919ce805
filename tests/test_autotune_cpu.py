"""The autotuner's choice on the host, with made-up times: the library's own choice by size is
among what it tries by default, is kept where it is the fastest, and is what a later call gets
from the cache; no candidate is the tile factor alone."""
import pytest

import lpm_inputs as li
from paper_0912_3223_gb300 import autotune, lpm

torch = pytest.importorskip("torch")


class FakeSim:
    def __init__(self):
        self.ctx = "ctx"
        self.cfg = li.make_cfg0(n_particles=10, n_steps=10)
        self.launch, self.every, self.resets = (128, 1, 0), 30, 0

    def reset(self):
        self.resets += 1


@pytest.fixture
def times(monkeypatch, tmp_path):
    """Times by (launch, interval), missing ones 9 ms; records what was timed."""
    sim, table, tried = FakeSim(), {}, []

    def set_auto(ctx, launch=True, sort=True):
        sim.launch = None if launch else sim.launch
        sim.every = None if sort else sim.every

    def time_shape(s, shape, reps=2):
        autotune._set_launch(s, shape)
        tried.append((s.launch, s.every))
        return table.get((s.launch, s.every), 9.0)

    monkeypatch.setenv("LPM_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "gpu")
    monkeypatch.setattr(lpm, "lpm_set_auto", set_auto)
    monkeypatch.setattr(lpm, "lpm_set_launch", lambda ctx, *s: setattr(sim, "launch", s))
    monkeypatch.setattr(lpm, "lpm_set_sort", lambda ctx, e: setattr(sim, "every", e))
    monkeypatch.setattr(autotune, "time_shape", time_shape)
    return sim, table, tried


@pytest.mark.parametrize("best", [None, (256, 1, 1)])
def test_launch(times, best):
    sim, table, tried = times
    table[best, 30] = 1.0
    assert autotune.autotune(sim) == best and sim.launch == best and sim.every == 30
    assert (None, 30) in tried and len(set(tried)) == len(tried) == 10
    sim.launch = (512, 1, 2)
    assert autotune.autotune(sim) == best and sim.launch == best and len(tried) == 10


@pytest.mark.parametrize("best", [(None, None), ((512, 1, 2), 120), (None, 0)])
def test_launch_and_sort(times, best):
    sim, table, tried = times
    table[best] = 1.0
    shape, every, ms = autotune.autotune_with_sort(sim)
    assert (shape, every) == best == (sim.launch, sim.every)
    assert (None, None) in tried and len(ms) == len(tried) == 10 * 6
    sim.launch, sim.every = (512, 1, 2), 60
    assert autotune.autotune_with_sort(sim)[:2] == best == (sim.launch, sim.every)
    assert len(tried) == 60


def test_given_candidates_only(times):
    sim, table, tried = times
    table[None, None] = 1.0
    table[(512, 1, 2), 60] = 2.0
    got = autotune.autotune_with_sort(sim, shapes=[(128, 1, 2), (512, 1, 2)], sort_intervals=(20, 60))
    assert got[:2] == ((512, 1, 2), 60) and len(got[2]) == 4
