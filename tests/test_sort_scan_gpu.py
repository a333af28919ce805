"""The sort's scan of key counts: weather grids whose number of sort keys lies at, just below
and above multiples of a scan tile (4096 keys) and beyond the tiles that a block adds up
itself, with whole-cell and cell-tile keys. Sorted runs give the unsorted run's results bit
for bit, also with counts left over from a sort and a changed interval in between."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu


def _cfg(nx, ny, nz, n, steps=40):
    base = li.make_cfg0(n_particles=n, n_steps=steps, kh=2000.0, kz=30.0)
    uvwk, z = li.make_artificial_weather(nx=nx, ny=ny, nz=nz, u=4.0, v=1.0, kz=30.0)
    # every grid spans the same 10 km around the source
    return dataclasses.replace(base, nx=nx, ny=ny, nz=nz, x0=-1000.0, y0=-5000.0,
                               dx=10000.0 / (nx - 1), dy=10000.0 / (ny - 1), z_levels=z,
                               uvwk=uvwk, lateral_exit=1, vd_dry=0.05, h_mix=200.0)


def _run(cfg, pieces, sort):
    from paper_0912_3223_gb300 import Sim
    from paper_0912_3223_gb300 import lpm
    with Sim(cfg, sort_every=sort[0]) as sim:
        for i, n in enumerate(pieces):
            if i and len(sort) > 1:
                lpm.lpm_set_sort(sim.ctx, sort[1])
            sim.step(n)
        xyz, tag = sim.particles()
        conc, dep, ctr, _ = sim.fixed_state()
    return xyz, tag, conc, dep, ctr


# keys = padded cells of whole 4 x 4 x 4 tiles, plus one for the dead
@pytest.mark.parametrize("nx,ny,nz,n", [
    (2, 2, 2, 3000),          # one cell tile
    (64, 60, 4, 140000),      # 15360 + 1 keys
    (64, 64, 4, 140000),      # 16384 + 1: the dead key alone in the last scan tile
    (63, 61, 3, 140000),
    (64, 64, 4, 5000),        # the same with cell-tile keys: 256 + 1
    (260, 252, 5, 140000),
    (1400, 1500, 8, 140000),  # 16.8e6 keys: more scan tiles than a block adds up
])
def test_sorted_runs_equal_unsorted(nx, ny, nz, n):
    cfg = _cfg(nx, ny, nz, n)
    ref = _run(cfg, [40], (0,))
    assert (ref[1] >> 28 == 2).any()             # some deposited
    for pieces, sort in (([40], (7,)), ([21, 19], (7, 3)), ([14, 14, 12], (14,))):
        for a, b in zip(ref, _run(cfg, pieces, sort)):
            assert np.array_equal(a, b)
