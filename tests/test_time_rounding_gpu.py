"""The advance step's time within the weather, bit for bit, where the first hour is not at 0
and steps are no binary fractions: t_k and its difference from the first hour's time are
rounded one by one in every instantiation and launch shape. Paths in a wind that changes with
time alone, and the rain hour of steps where one rounding instead of two picks another hour."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

F = np.float32
STEPS = 130


def _since(cfg, k):
    return F(F(F(k) * F(cfg.dt)) - F(cfg.met_t0))


def _path(cfg, k0):
    """FP32 x and y of a particle released at step k0 (no diffusion; fused multiply-adds)."""
    a, b = cfg.uvwk[:, 0, 0, 0, :2]
    x = np.array([cfg.src_x, cfg.src_y], F)
    for k in range(k0, cfg.n_steps):
        ft = F(_since(cfg, k) * F(1.0 / cfg.met_dt))
        f = np.float64(min(max(ft, F(0.0)), F(1.0)))
        u = (f * (b - a).astype(np.float64) + a).astype(F)
        x = (u.astype(np.float64) * np.float64(F(cfg.dt)) + x).astype(F)
    return x


def _config(dt, t0, n):
    base = li.make_cfg0(n_particles=n, n_steps=STEPS, kh=0.0, kz=0.0)
    uvwk = np.zeros_like(base.uvwk)
    uvwk[0, ..., :2], uvwk[1, ..., :2] = (1.3, -0.7), (4.9, 2.1)
    return dataclasses.replace(base, uvwk=uvwk, dt=dt, met_t0=t0, met_dt=5000.0)


@pytest.mark.parametrize("dt,t0", [(33.1, 345.6), (7.3, 7.77), (33.1, -1234.5)])
@pytest.mark.parametrize("kind", ["plain", "drift", "langevin", "dosage", "ensemble"])
@pytest.mark.parametrize("launch,sort_every", [(None, None), ((256, 1, 1), 0), ((512, 1, 2), 30)])
def test_paths(dt, t0, kind, launch, sort_every):
    from paper_0912_3223_gb300 import Sim
    cfg = _config(dt, t0, STEPS)
    if kind == "drift":
        cfg = dataclasses.replace(cfg, drift_correction=1)
    if kind == "langevin":
        cfg = dataclasses.replace(cfg, langevin=1, t_lagr=50.0)
    if kind == "ensemble":
        scen = [li.Scenario(cfg.src_x, cfg.src_y, cfg.src_z, cfg.release) for _ in range(2)]
        cfg = dataclasses.replace(cfg, n_scenarios=2, scenarios=scen)
    want = np.array([_path(cfg, k) for k in range(STEPS)])      # particle k leaves at step k
    with Sim(cfg, launch=launch, sort_every=sort_every) as sim:
        if kind == "dosage":
            sim.set_dosage(7)
        sim.step(STEPS)
        got = sim.particles()[0][:, :2]
    for g in np.split(got, len(got) // STEPS):
        assert np.array_equal(g, want)


@pytest.mark.parametrize("k", [7, 14, 63, 66])
@pytest.mark.parametrize("langevin", [0, 1])
@pytest.mark.parametrize("launch", [None, (256, 1, 1), (512, 1, 2)])
def test_rain_hour(k, langevin, launch):
    from paper_0912_3223_gb300 import Sim
    T = 33.1                                      # step, hour and the first hour's time
    base = _config(T, T, 64)
    hour = int(np.floor(F(_since(base, k) / F(T))))
    once = np.floor(F(np.float64(F(k)) * np.float64(F(T)) - np.float64(F(T))) / F(T))
    assert hour != once                           # one rounding less is another hour
    rain = np.zeros((70, base.ny, base.nx), np.uint8)
    rain[hour] = 1
    cfg = dataclasses.replace(base, n_met_t=70, met_dt=T, uvwk=np.repeat(base.uvwk[:1], 70, 0),
                              rain=rain, wet_lambda=10.0, langevin=langevin, t_lagr=50.0,
                              release=li.Release(64, np.array([1.0]), 3600.0, k, k + 1))
    with Sim(cfg, launch=launch) as sim:
        sim.step(k + 1)
        tag = sim.particles()[1]
    assert (tag >> 28 == li.STATUS_DEP_WET).all()
