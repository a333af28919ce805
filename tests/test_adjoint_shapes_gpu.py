"""The adjoint's segment kernels at the sizes where their launch shape and groups change: one
particle, a group of 128 less and more than full, segments on both sides of the few-groups
rule (4 groups of 128 an SM: 77824 particles on 152 SMs), scenarios whose groups share a
block, uniform and gridded K_h. The sorted forms agree with the release-order form (whose
kernels are others) and with each other to the roundings that they may differ by."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

SIGMA, EVERY, STEPS = 200.0, 9, 150            # three segments, the last one partial


def _forms(cfg, n_scen):
    from paper_0912_3223_gb300 import Sim, lpm
    rec = li.make_receptors(down=(300.0, 6000.0), cross=1500.0)
    w = np.linspace(-1.0, 1.0, n_scen * rec.shape[0]).reshape(n_scen, -1)
    out = {}
    for form, limit, sort in (("trajectory", 1 << 37, 60), ("checkpoints", 0, 60),
                              ("release order", 1 << 37, 0)):
        with Sim(cfg, sort_every=sort) as sim:
            lpm.lpm_set_adjoint_storage(sim.ctx, limit)
            C = lpm.lpm_receptors(sim.ctx, n_scen, rec, SIGMA, EVERY)
            out[form] = C, lpm.lpm_adjoint(sim.ctx, rec, SIGMA, EVERY, w, 24)
    return out


def _compare(out):
    C0, g0 = out["release order"]
    C1, g1 = out["trajectory"]
    C2, g2 = out["checkpoints"]
    assert np.abs(C0).max() > 0
    # the same FP32 terms in FP64 sums of another order
    for C in (C1, C2):
        np.testing.assert_allclose(C, C0, rtol=1e-12, atol=1e-15 * np.abs(C0).max())
    np.testing.assert_allclose(g2, g1, rtol=1e-9, atol=1e-12 * np.abs(g1).max())
    np.testing.assert_allclose(g1[:, :3], g0[:, :3], rtol=1e-9, atol=1e-12 * np.abs(g0[:, :3]).max())
    # a particle's FP32 parameter sums restart every 64 steps in the sorted forms
    np.testing.assert_allclose(g1[:, 3:], g0[:, 3:], rtol=0, atol=2e-5 * np.abs(g0[:, 3:]).max())


@pytest.mark.parametrize("n", [1, 127, 129, 77000, 79000])
@pytest.mark.parametrize("gridded_kh", [False, True])
def test_one_release(n, gridded_kh):
    cfg = li.make_cfg3(n_particles=n, n_steps=STEPS)
    # everything leaves in the first 60 steps: later segments hold all that still moves
    cfg = dataclasses.replace(cfg, release=dataclasses.replace(cfg.release, last_step=60))
    if gridded_kh:
        kh = np.random.default_rng(3).uniform(50.0, 150.0, cfg.uvwk.shape[:4]).astype(np.float32)
        cfg = dataclasses.replace(cfg, kh=kh, kh_uniform=-1.0)
    _compare(_forms(cfg, 1))


@pytest.mark.parametrize("counts", [(130, 127, 1, 300), (30000, 129, 50000)])
def test_scenarios(counts):
    base = li.make_cfg3(n_particles=1, n_steps=STEPS)
    scen = [li.Scenario(5000.0 + 100.0 * s, 24875.0 - 150.0 * s, 40.0 + 10.0 * s,
                        li.Release(n, base.release.q, 3600.0, 0, 60))
            for s, n in enumerate(counts)]
    cfg = dataclasses.replace(base, n_scenarios=len(scen), scenarios=scen)
    _compare(_forms(cfg, len(scen)))
