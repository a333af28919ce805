"""The launch shape that the library picks by size and options gives the results of a fixed
shape bit for bit: particle counts around a warp, the tile sizes, the limits of the shapes'
ranges (20 warps an SM: 97280 particles on 152 SMs; 8 times that), with and without the sorts
(launches longer than a step table are cut), for the plain step, the options and an ensemble."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS = 135                                    # past a table of 128 steps and two sorts


def _run(cfg, launch, sort_every):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch, sort_every=sort_every) as sim:
        if getattr(cfg, "dosage_every", 0):
            sim.set_dosage(cfg.dosage_every)
        sim.step(cfg.n_steps)
        xyz, tag = sim.particles()
        fixed = [sim.fixed_state(s)[:3] for s in range(cfg.n_scenarios)]
    return xyz, tag, fixed


def _same(a, b):
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for x, y in zip(a[2], b[2]):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)


@pytest.mark.parametrize("n", [1, 31, 33, 513, 19456, 19457, 97280, 97281, 131072, 131073, 778241])
@pytest.mark.parametrize("sort_every", [60, 0])
def test_plain_sizes(n, sort_every):
    cfg = dataclasses.replace(li.make_cfg0(n_particles=n, n_steps=STEPS), half_life_s=3600.0)
    auto = _run(cfg, None, sort_every)
    _same(auto, _run(cfg, (512, 1, 2), sort_every))
    if n in (33, 97281):
        _same(auto, _run(cfg, (128, 4, 1), sort_every))


@pytest.mark.parametrize("n", [33, 97281, 131073])
def test_extended_step(n):
    cfg = dataclasses.replace(li.make_cfg0(n_particles=n, n_steps=STEPS), langevin=1, t_lagr=50.0)
    cfg.dosage_every = 7
    _same(_run(cfg, None, 60), _run(cfg, (512, 1, 2), 60))


@pytest.mark.parametrize("n_min,n_max,scenarios", [(1, 40, 5), (2000, 9000, 20), (30000, 60000, 4)])
def test_ensemble(n_min, n_max, scenarios):
    cfg = li.make_cfg2(n_scenarios=scenarios, n_steps=STEPS, n_min=n_min, n_max=n_max)
    _same(_run(cfg, None, 60), _run(cfg, (512, 1, 2), 60))
