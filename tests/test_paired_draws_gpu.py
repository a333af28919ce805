"""Small runs, where one warp of a pair draws for the other, give the results of a fixed launch
shape bit for bit: particle counts around a warp and around the limit of the rule (8 warps an
SM: 38912 particles on 152 SMs), calls of 1 to 9 steps (parts of a buffer of 4 steps, odd first
steps), releases in the middle of a launch, particles that all stop early, every instantiation."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

PIECES = (1, 2, 3, 4, 5, 6, 7, 8, 9, 100, 1)


def _run(cfg, launch, sort_every, pieces):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch, sort_every=sort_every) as sim:
        for n in pieces:
            sim.step(n)
        xyz, tag = sim.particles()
        fixed = [sim.fixed_state(s)[:3] for s in range(cfg.n_scenarios)]
    return [xyz, tag] + [a for f in fixed for a in f]


def _same(cfg, pieces=PIECES, sort_every=None):
    a = _run(cfg, None, sort_every, pieces)
    b = _run(cfg, (512, 1, 2), 0, pieces)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    return a


def _plain(n, **kw):
    cfg = li.make_cfg3(n_particles=n, n_steps=sum(PIECES))
    return dataclasses.replace(cfg, bin_every=20, **kw)


@pytest.mark.parametrize("n", [1, 31, 33, 4097, 38880, 38912, 38913])
def test_sizes(n):
    _same(_plain(n))


@pytest.mark.parametrize("first,last", [(0, 1), (3, 4), (7, 90), (145, 146)])
def test_releases(first, last):
    cfg = _plain(500)
    _same(dataclasses.replace(cfg, release=dataclasses.replace(cfg.release, first_step=first,
                                                               last_step=last)))


@pytest.mark.parametrize("vd", [0.0, 30.0])
def test_no_deposition_and_all_stopped(vd):
    cfg = _plain(3000, vd_dry=vd, h_mix=100000.0, wet_lambda=0.0)
    cfg = dataclasses.replace(cfg, release=dataclasses.replace(cfg.release, last_step=2))
    # at 30 m/s and 100 km a step of 20 s deposits 0.6 %; at 1 km, 60 %
    _same(cfg)
    tag = _same(dataclasses.replace(cfg, h_mix=1000.0))[1]
    if vd > 0:
        assert ((tag >> 28) != 0).mean() > 0.9


@pytest.mark.parametrize("drift", [0, 1])
@pytest.mark.parametrize("n_modes", [0, 3])
@pytest.mark.parametrize("sort_every", [None, 25])
def test_ensemble(drift, n_modes, sort_every):
    cfg = li.make_cfg2(n_scenarios=7, n_steps=sum(PIECES), n_min=30, n_max=4000, n_modes=n_modes)
    _same(dataclasses.replace(cfg, drift_correction=drift, bin_every=20), sort_every=sort_every)


def test_drift_of_one_scenario():
    _same(_plain(2001, drift_correction=1), sort_every=30)
