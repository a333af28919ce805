"""The weather records' order (lines of 2 rows x 2 levels, each lane of a group of four
loading a cell's corners in an order of its own) on grids with odd and smallest sizes: one
step without diffusion moves every particle by the 4D-linear wind at its source, whatever
lane it sits in, in release order and sorted. Sources at nodes, cell centres, edges and
outside the grid; compared with FP64 interpolation in numpy."""
import dataclasses

import numpy as np
import pytest

import lpm_inputs as li

pytestmark = pytest.mark.gpu

DT, SPACING, LANES = 10.0, 250.0, 7


def _interp(cfg, field, x, y, z):
    """Multilinear value of field [nz][ny][nx] at a point (constant beyond the grid)."""
    def axis(v, nodes):
        i = int(np.clip(np.searchsorted(nodes, v, side="right") - 1, 0, len(nodes) - 2))
        return i, float(np.clip((v - nodes[i]) / (nodes[i + 1] - nodes[i]), 0.0, 1.0))
    i, a = axis(x, np.arange(cfg.nx) * SPACING)
    j, b = axis(y, np.arange(cfg.ny) * SPACING)
    k, c = axis(z, np.asarray(cfg.z_levels))
    f = field[k:k + 2, j:j + 2, i:i + 2].astype(np.float64)
    wx, wy, wz = np.array([1 - a, a]), np.array([1 - b, b]), np.array([1 - c, c])
    return float(np.einsum("kji,k,j,i", f, wz, wy, wx))


@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 2), (3, 2, 2), (2, 3, 2), (2, 2, 3), (5, 4, 3),
                                      (4, 5, 6), (7, 7, 7)])
@pytest.mark.parametrize("gridded_kh", [False, True])
@pytest.mark.parametrize("sort_every", [0, 1])
def test_one_step_follows_the_interpolated_wind(nx, ny, nz, gridded_kh, sort_every):
    from paper_0912_3223_gb300 import Sim
    rng = np.random.default_rng(100 * nx + 10 * ny + nz)
    base = li.make_cfg0(n_particles=1, n_steps=2, kh=0.0, kz=0.0)
    z_levels = 40.0 * np.arange(nz) + 10.0
    uvwk = np.zeros((2, nz, ny, nx, 4), np.float32)
    uvwk[..., :3] = rng.uniform(-4.0, 4.0, (2, nz, ny, nx, 3))
    # a gridded K_h that vanishes: its code runs and adds nothing
    kh = np.zeros((2, nz, ny, nx), np.float32) if gridded_kh else None
    lx, ly = (nx - 1) * SPACING, (ny - 1) * SPACING
    pts = [(0.0, 0.0, 10.0), (lx, ly, z_levels[-1]), (-300.0, ly / 2, 30.0),
           (lx / 2, ly + 400.0, 5.0 + z_levels[-1]), (lx / 2, ly / 2, 2.0)]
    pts += [(SPACING * (i + 0.5), SPACING * (j + 0.25), z_levels[k] + 17.0)
            for i in range(nx - 1) for j in range(ny - 1) for k in range(nz - 1)][:40]
    # sources that single precision holds exactly
    pts = [tuple(float(np.float32(v)) for v in p) for p in pts]
    scen = [li.Scenario(*p, li.Release(LANES, np.array([1.0]), 3600.0, 0, 1)) for p in pts]
    cfg = dataclasses.replace(base, nx=nx, ny=ny, nz=nz, x0=0.0, y0=0.0, dx=SPACING, dy=SPACING,
                              z_levels=z_levels, uvwk=uvwk, kh=kh, dt=DT,
                              kh_uniform=-1.0 if gridded_kh else 0.0, reflect_ground=0,
                              n_scenarios=len(scen), scenarios=scen, bin_every=2)
    with Sim(cfg, sort_every=sort_every) as sim:
        sim.step(1)
        one = sim.particles()[0].astype(np.float64).reshape(len(pts), LANES, 3)
        sim.step(1)
        two = sim.particles()[0].astype(np.float64).reshape(len(pts), LANES, 3)
    assert np.ptp(one, axis=1).max() == 0.0 and np.ptp(two, axis=1).max() == 0.0
    f = np.float64(DT) / 3600.0                    # the second step's fraction of the hour
    # roundings of one step, each half an ulp (2^-24 relative): fractions of up to 8 cells' width
    # (position, difference, product: 3 x 2^-24 x 8), eight blends of |u| <= 4 in four levels
    # (each a difference of up to 8 and a product: 3 x 8 x 2^-24 x 4 levels), the move
    # (3 roundings of |x| <= 2500); the fractions' error acts on differences of up to 8
    eps = 2.0 ** -24
    tol = eps * (DT * (8 * 3 * 8 * 3 + 3 * 8 * 4) + 3 * 2500.0)
    for s, p in enumerate(pts):
        u0 = [_interp(cfg, uvwk[0, ..., q], *p) for q in range(3)]
        want = np.asarray(p) + DT * np.asarray(u0)
        assert np.abs(one[s, 0] - want).max() <= tol, (p, one[s, 0], want)
        w = (1 - f) * uvwk[0].astype(np.float64) + f * uvwk[1]
        u1 = [_interp(cfg, w[..., q], *one[s, 0]) for q in range(3)]
        want = one[s, 0] + DT * np.asarray(u1)
        assert np.abs(two[s, 0] - want).max() <= tol, (p, two[s, 0], want)
