"""The sort interval that the library picks by size gives the results of fixed ones bit for bit:
at the limits of its ranges (65536 and 2^20 particles, 2^19 with the extended step), for an
ensemble, and where an option that is switched on during the run changes the interval."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS = 250                                    # past two sorts of 120 steps


def _run(cfg, sort_every, dosage_from=None):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, sort_every=sort_every) as sim:
        if dosage_from is not None:
            sim.step(dosage_from)
            sim.set_dosage(10)
            sim.step(cfg.n_steps - dosage_from)
        else:
            sim.step(cfg.n_steps)
        xyz, tag = sim.particles()
        fixed = [sim.fixed_state(s)[:3] for s in range(cfg.n_scenarios)]
    return [xyz, tag] + [a for f in fixed for a in f]


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n", [65536, 65537, 1 << 20, (1 << 20) + 1])
def test_plain_limits(n):
    cfg = dataclasses.replace(li.make_cfg0(n_particles=n, n_steps=STEPS), half_life_s=3600.0)
    auto = _run(cfg, None)
    _same(auto, _run(cfg, 60))
    _same(auto, _run(cfg, 0))


@pytest.mark.parametrize("n", [1 << 19, (1 << 19) + 1])
def test_extended_limits(n):
    cfg = dataclasses.replace(li.make_cfg0(n_particles=n, n_steps=STEPS), langevin=1, t_lagr=50.0)
    _same(_run(cfg, None), _run(cfg, 60))


@pytest.mark.parametrize("scenarios,n", [(3, 4000), (7, 40000)])
def test_ensemble(scenarios, n):
    cfg = li.make_cfg2(n_scenarios=scenarios, n_steps=STEPS, n_min=n // 2, n_max=n)
    _same(_run(cfg, None), _run(cfg, 60))


@pytest.mark.parametrize("at", [60, 130])
def test_interval_changes_during_the_run(at):
    # 120 steps between sorts without the dosage samples, 60 with them
    cfg = li.make_cfg0(n_particles=600000, n_steps=STEPS)
    _same(_run(cfg, None, at), _run(cfg, 60, at))
