"""The read-backs through the C ABI: after a device error they report it and leave every array
of the caller as it was; otherwise each output alone is what the whole call gives."""
import ctypes as C
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

PLANE, CELLS, N = (13, 17), (5, 13, 17), 3001
F64, U64, F32, U32, I64 = (C.POINTER(t) for t in (C.c_double, C.c_uint64, C.c_float,
                                                  C.c_uint32, C.c_int64))


def _config(**kw):
    base = li.make_cfg1(n_particles=N, n_steps=40, n_hours=2)
    return dataclasses.replace(base, cx=17, cy=13, cz=5, cdx=4000.0, cdy=4000.0, cdz=500.0,
                               bin_every=20, vd_dry=0.3, langevin=1, t_lagr=100.0,
                               chain_half_lives=np.array([base.half_life_s, 3600.0, 0.0]), **kw)


def _calls(L, ctx):
    """(call, output arrays by their types) of every read-back."""
    cells, plane = int(np.prod(CELLS)), int(np.prod(PLANE))
    v = C.c_void_p(ctx)
    return {
        "concentration": (lambda a: L.lpm_concentration(v, 0, a, cells), [(F64, CELLS)]),
        "deposition": (lambda a, b: L.lpm_deposition(v, 0, a, b, plane), [(F64, PLANE)] * 2),
        "budget": (lambda a: L.lpm_budget(v, 0, a), [(F64, 8)]),
        "particles": (lambda a, b: L.lpm_particles(v, 0, N, a, b), [(F32, (N, 3)), (U32, N)]),
        "velocity": (lambda a: L.lpm_particle_velocity(v, 0, N, a), [(F32, N)]),
        "fixed_state": (lambda a, b, c: L.lpm_fixed_state(v, 0, a, cells, b, 2 * plane, c, None),
                        [(U64, CELLS), (U64, (2,) + PLANE), (I64, 16)]),
        "species": (lambda a, b, c, d, e: L.lpm_species(v, 0, 1, a, b, c, d, e),
                    [(F64, CELLS), (F64, PLANE), (F64, PLANE), (U64, CELLS), (U64, (2,) + PLANE)]),
        "dosage": (lambda a, b, c: L.lpm_dosage(v, 0, a, cells, b, c),
                   [(F64, CELLS), (U64, CELLS), (I64, 1)]),
    }


def _arrays(outs):
    a = [np.empty(shape, dtype=t._type_) for t, shape in outs]
    for x in a:
        x.view(np.uint8)[...] = 0xA5
    return a


def _args(arrays, outs, keep):
    return [x.ctypes.data_as(t) if i in keep else None for i, (x, (t, _)) in
            enumerate(zip(arrays, outs))]


@pytest.mark.parametrize("sort_every", [None, 10])
def test_an_error_leaves_the_arrays(sort_every):
    from paper_0912_3223_gb300 import Sim, lpm
    cfg = _config()
    bad = cfg.uvwk.copy()
    bad[..., 0] = np.nan
    with Sim(dataclasses.replace(cfg, uvwk=bad), sort_every=sort_every) as sim:
        sim.set_dosage(5)
        sim.step(40)
        for name, (call, outs) in _calls(lpm.load(), sim.ctx).items():
            arrays = _arrays(outs)
            assert call(*_args(arrays, outs, range(len(outs)))) == lpm.LPM_E_NUMERIC, name
            for x in arrays:
                assert (x.view(np.uint8) == 0xA5).all(), name


@pytest.mark.parametrize("sort_every", [None, 10])
def test_single_outputs(sort_every):
    from paper_0912_3223_gb300 import Sim, lpm
    with Sim(_config(), sort_every=sort_every) as sim:
        sim.set_dosage(5)
        sim.step(40)
        for name, (call, outs) in _calls(lpm.load(), sim.ctx).items():
            whole = _arrays(outs)
            assert call(*_args(whole, outs, range(len(outs)))) == lpm.LPM_OK, name
            if len(outs) == 1:
                continue
            for keep in range(len(outs)):
                arrays = _arrays(outs)
                assert call(*_args(arrays, outs, [keep])) == lpm.LPM_OK, name
                for i, (x, w) in enumerate(zip(arrays, whole)):
                    if i == keep:
                        assert np.array_equal(x, w), (name, keep)
                    else:
                        assert (x.view(np.uint8) == 0xA5).all(), (name, keep)


def test_without_room_on_the_device():
    """On a full device the read-backs convert on the host and give the same bits."""
    import torch
    from paper_0912_3223_gb300 import Sim
    cfg = dataclasses.replace(_config(release=li.Release(5_000_000, np.array([1.0]), 3600.0, 0, 2)),
                              cx=400, cy=400, cz=60, cdx=125.0, cdy=125.0, cdz=50.0, n_steps=4,
                              bin_every=2, langevin=0)
    need = 4 * min(cfg.n_particles, 1 << 22) * 4          # the smaller of the two scratches

    def outputs(sim):
        return [*sim.particles(), sim.concentration(), *sim.deposition(), *sim.species(1),
                *sim.dosage()[:2]]

    sims = [Sim(cfg, sort_every=0).set_dosage(2).step(4) for _ in range(2)]
    want = outputs(sims[0])                               # (loads the kernels, too)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (32 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < need
        got = outputs(sims[1])
    finally:
        del fill
        torch.cuda.empty_cache()
        for sim in sims:
            sim.close()
    assert want[2].max() > 0 and want[8].max() > 0
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
