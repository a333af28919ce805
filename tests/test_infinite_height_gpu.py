"""A source at an infinite height (a double beyond single precision, or lpm_create's source,
which is not checked) samples the top cell of the weather as one far above it does: the cell
lookup has no level above the top cell. Both give the same bits where the reflections bring
the particles back to the model top, and an infinite position is reported where nothing does.
Every place that the level entries are read from, with odd and even numbers of levels."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

STEPS, FAR = 9, 1e38


def _config(nz, z_src, n=70, **kw):
    base = li.make_cfg0(n_particles=n, n_steps=STEPS)
    rng = np.random.default_rng(nz)
    uvwk = rng.uniform(0.5, 4.0, (2, nz, 5, 4, 4)).astype(np.float32)
    cfg = dataclasses.replace(base, nx=4, ny=5, nz=nz, dx=2000.0, dy=2000.0, uvwk=uvwk,
                              z_levels=100.0 * np.arange(nz), reflect_top=1,
                              z_top=100.0 * (nz - 1), src_z=z_src)
    return dataclasses.replace(cfg, **kw)


def _options(kind, nz):
    kh = np.random.default_rng(1).uniform(20.0, 60.0, (2, nz, 5, 4)).astype(np.float32)
    return {"plain": {}, "kh": dict(kh=kh, kh_uniform=-1.0), "drift": dict(drift_correction=1),
            "langevin": dict(langevin=1, t_lagr=50.0)}[kind]


def _run(cfg, launch, sort_every):
    from paper_0912_3223_gb300 import Sim
    with Sim(cfg, launch=launch, sort_every=sort_every) as sim:
        sim.step(STEPS)
        xyz, tag = sim.particles()
        conc, dep, ctr, _ = sim.fixed_state()
    return xyz, tag, conc, dep, ctr


@pytest.mark.parametrize("nz", [2, 3, 6, 7])
@pytest.mark.parametrize("kind", ["plain", "kh", "drift", "langevin"])
@pytest.mark.parametrize("launch,sort_every", [(None, None), ((256, 1, 0), 0), ((512, 1, 2), 3)])
def test_reflected(nz, kind, launch, sort_every):
    kw = _options(kind, nz)
    far = _run(_config(nz, FAR, **kw), launch, sort_every)
    assert np.isfinite(far[0]).all() and np.ptp(far[0][:, 2]) > 0
    for z in (np.inf, 1e39):
        for a, b in zip(_run(_config(nz, z, **kw), launch, sort_every), far):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("nz", [6, 7])
@pytest.mark.parametrize("limit", [1 << 37, 0])
@pytest.mark.parametrize("sort_every", [None, 0])
def test_receptors(nz, limit, sort_every):
    from paper_0912_3223_gb300 import Sim, lpm
    rec = np.array([[0.0, 0.0, 50.0], [100.0, 50.0, 100.0 * (nz - 1)]])
    out = []
    for z in (FAR, np.inf):
        with Sim(_config(nz, z), sort_every=sort_every) as sim:
            lpm.lpm_set_adjoint_storage(sim.ctx, limit)
            out.append(lpm.lpm_receptors(sim.ctx, 1, rec, 200.0, 3))
    assert out[0].max() > 0
    # the same FP32 terms in FP64 sums whose order may differ
    np.testing.assert_allclose(out[1], out[0], rtol=1e-12)


@pytest.mark.parametrize("nz", [6, 7])
def test_not_reflected(nz):
    from paper_0912_3223_gb300 import Sim, lpm
    cfg = _config(nz, np.inf, reflect_top=0, z_top=0.0)
    with Sim(cfg) as sim:
        sim.step(1)
        with pytest.raises(lpm.LpmError) as e:
            sim.sync()
    assert e.value.status == lpm.LPM_E_NUMERIC
