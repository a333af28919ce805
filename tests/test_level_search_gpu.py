"""Levels too narrow for the lookup table (bisection) give the results of levels with one:
both grids share every level up to z_top, where the particles stay, and differ above it by a
level 0.25 m over another. The step in every option's instantiation and launch shape, and the
receptor sweeps, whose cells are looked up in the same tables."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS = 70                                     # a sort in between


def _extend(cfg, narrow):
    """`cfg` with more levels above its top, `narrow`: two of them 0.25 m apart."""
    z = np.asarray(cfg.z_levels, dtype=np.float64)
    top = float(z[-1])
    more = [top + 512.0] + ([top + 512.25] if narrow else []) + [top + 1024.0]

    def up(a, axis):
        return np.concatenate([a] + [np.take(a, [-1], axis)] * len(more), axis)

    kw = dict(nz=len(z) + len(more), z_levels=np.concatenate([z, more]), uvwk=up(cfg.uvwk, 1),
              reflect_top=1, z_top=top)
    if cfg.kh is not None:
        kw["kh"] = up(cfg.kh, 1)
    if cfg.modes is not None:
        kw["mode_profile"] = up(np.asarray(cfg.mode_profile), 0)
    return dataclasses.replace(cfg, **kw)


def _run(cfg, launch, dosage):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch) as sim:
        if dosage:
            sim.set_dosage(dosage)
        sim.step(cfg.n_steps)
        xyz, tag = sim.particles()
        fixed = [sim.fixed_state(s)[:3] for s in range(cfg.n_scenarios)]
    return [xyz, tag] + [a for f in fixed for a in f]


def _config(kind):
    if kind.startswith("modes"):
        cfg = li.make_cfg2(n_scenarios=3, n_steps=STEPS, n_min=1000, n_max=5000)
    else:
        cfg = li.make_cfg3(n_particles=5003, n_steps=STEPS)
    if kind.endswith("drift"):
        cfg = dataclasses.replace(cfg, drift_correction=1)
    if kind == "langevin":
        cfg = dataclasses.replace(cfg, langevin=1, t_lagr=50.0)
    return cfg


@pytest.mark.parametrize("kind", ["plain", "drift", "modes", "modes drift", "langevin", "dosage"])
@pytest.mark.parametrize("launch", [None, (256, 1, 1), (512, 1, 2)])
def test_step(kind, launch):
    cfg = _config(kind)
    dosage = 7 if kind == "dosage" else 0
    a = _run(_extend(cfg, False), launch, dosage)
    b = _run(_extend(cfg, True), launch, dosage)
    assert np.ptp(a[0][:, 2]) > 0
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("scenarios", [1, 3])
@pytest.mark.parametrize("sort_every", [60, 0])
@pytest.mark.parametrize("limit", [1 << 37, 0])
def test_receptor_sweeps(scenarios, sort_every, limit):
    from paper_0912_3223_gb300 import Sim, lpm
    cfg = li.make_cfg3(n_particles=5003, n_steps=STEPS)
    if scenarios > 1:
        scen = [li.Scenario(5000.0 + 100.0 * s, 24875.0 - 150.0 * s, 40.0 + 10.0 * s,
                            li.Release(1000 + 129 * s, cfg.release.q, 3600.0, 0, STEPS))
                for s in range(scenarios)]
        cfg = dataclasses.replace(cfg, n_scenarios=scenarios, scenarios=scen)
    rec = li.make_receptors(down=(300.0, 6000.0), cross=1500.0)
    w = np.linspace(-1.0, 1.0, scenarios * rec.shape[0]).reshape(scenarios, -1)
    out = []
    for narrow in (False, True):
        with Sim(_extend(cfg, narrow), sort_every=sort_every) as sim:
            lpm.lpm_set_adjoint_storage(sim.ctx, limit)
            C = lpm.lpm_receptors(sim.ctx, scenarios, rec, 200.0, 9)
            out.append((C, lpm.lpm_adjoint(sim.ctx, rec, 200.0, 9, w, 24)))
    # the same FP32 terms, the order of the FP64 sums aside
    (C0, g0), (C1, g1) = out
    assert np.abs(C0).max() > 0
    np.testing.assert_allclose(C1, C0, rtol=1e-12, atol=1e-15 * np.abs(C0).max())
    np.testing.assert_allclose(g1, g0, rtol=1e-9, atol=1e-12 * np.abs(g0).max())
