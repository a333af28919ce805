"""The launch shapes that the library picks on both sides of its limits (216 warps of particles an
SM, 75 for the extended step and for mixed scenarios, and 8 times those, above which one shape
is launched instead of two) give the results of a fixed shape bit for bit."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS = 20


def _run(cfg, launch):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch) as sim:
        sim.step(cfg.n_steps)
        xyz, tag = sim.particles()
        fixed = [sim.fixed_state(s)[:3] for s in range(cfg.n_scenarios)]
    return [xyz, tag] + [a for f in fixed for a in f]


def _same(cfg):
    for x, y in zip(_run(cfg, None), _run(cfg, (512, 1, 2))):
        assert np.array_equal(x, y)


def _particles(warps_per_sm):
    import torch
    return warps_per_sm * torch.cuda.get_device_properties(0).multi_processor_count * 32


@pytest.mark.parametrize("warps,more", [(216, 0), (216, 1), (8 * 216, 1)])
def test_plain(warps, more):
    _same(li.make_cfg0(n_particles=_particles(warps) + more, n_steps=STEPS))


@pytest.mark.parametrize("warps,more", [(75, 0), (75, 1), (216, 1), (8 * 75, 1)])
def test_extended(warps, more):
    _same(dataclasses.replace(li.make_cfg0(n_particles=_particles(warps) + more, n_steps=STEPS),
                              langevin=1, t_lagr=50.0))


@pytest.mark.parametrize("warps", [74, 76])
def test_ensemble(warps):
    n = _particles(warps)
    _same(li.make_cfg2(n_scenarios=4, n_steps=STEPS, n_min=n // 4, n_max=n // 4 + 1))
