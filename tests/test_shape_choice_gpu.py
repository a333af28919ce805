"""The launches of two shapes of which the device's count of live particles lets one run: after
a sort, fewer particles than the host's bound may still move. Each shape runs, at and around the
limits (216 warps of particles an SM, 75 for the extended step and for mixed scenarios), with the
bits of a fixed shape, active-step counters included. Eq. 3 and a decay chain on both sides of
the extended step's limits, too."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS, EVERY = 45, 20


def _warps(per_sm):
    import torch
    return per_sm * torch.cuda.get_device_properties(0).multi_processor_count


def _run(cfg, launch, dosage=0):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch, sort_every=EVERY) as sim:
        if dosage:
            sim.set_dosage(dosage)
        sim.step(EVERY)
        live = int((sim.particles()[1] >> 28 == li.STATUS_ACTIVE).sum())
        sim.step(cfg.n_steps - EVERY)
        out = [*sim.particles()]
        for s in range(cfg.n_scenarios):
            out += sim.fixed_state(s)[:3]
            if dosage:
                out.append(sim.dosage(s)[1])
            for j in range(1, 0 if cfg.chain_half_lives is None else 3):
                out += sim.species(j, s)[3:]
    return live, out


def _same(cfg, dosage=0):
    live, a = _run(cfg, None, dosage)
    _, b = _run(cfg, (512, 1, 2), dosage)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    return live


def _release(n):
    return li.Release(n, np.array([1.0]), 3600.0, 0, 2)


def _deposits(cfg):
    """5 % of the particles a step: about a third is left at the first sort."""
    return dataclasses.replace(cfg, vd_dry=5.0, h_mix=1000.0)


def test_plain():
    few = 32 * _warps(216)
    cfg = li.make_cfg0(n_particles=2 * few, n_steps=STEPS)
    live = _same(_deposits(dataclasses.replace(cfg, release=_release(2 * few))))
    assert 0 < live <= few - 32


@pytest.mark.parametrize("kind", ["langevin", "dosage"])
def test_extended(kind):
    few = 32 * _warps(75)
    cfg = _deposits(dataclasses.replace(li.make_cfg0(n_particles=2 * few, n_steps=STEPS),
                                        release=_release(2 * few)))
    if kind == "langevin":
        cfg = dataclasses.replace(cfg, langevin=1, t_lagr=50.0)
    live = _same(cfg, dosage=7 if kind == "dosage" else 0)
    assert 0 < live <= few - 32


@pytest.mark.parametrize("more", [-31, 0, 1, 40])
@pytest.mark.parametrize("langevin", [0, 1])
def test_ensemble_at_the_limit(more, langevin):
    """The first scenario stays, the second starts outside the domain and leaves at once: after
    the sort exactly the first one's particles are counted."""
    stay = 32 * _warps(75) + more
    base = li.make_cfg0(n_particles=1, n_steps=STEPS)
    scen = [li.Scenario(0.0, 0.0, 50.0, _release(stay)),
            li.Scenario(0.0, 9000.0, 50.0, _release(40000))]
    cfg = dataclasses.replace(base, n_scenarios=2, scenarios=scen, lateral_exit=1,
                              langevin=langevin, t_lagr=50.0)
    assert _same(cfg) == stay


@pytest.mark.parametrize("per_sm,more", [(75, 0), (75, 1), (216, 1)])
def test_eq3_and_chain(per_sm, more):
    n = 32 * _warps(per_sm) + more
    cfg = li.make_cfg1(n_particles=n, n_steps=EVERY + 5, n_hours=2, kz_eq3=True)
    cfg = dataclasses.replace(cfg, release=_release(n),
                              chain_half_lives=np.array([cfg.half_life_s, 3600.0, 0.0]))
    _same(cfg)
