"""Performance cases of the particle model: what its users have it compute, through the
public entry points (`Sim`, `receptor_concentrations`, `invert`).

A case names a form and its sizes:

  plain      one release: reset, all steps, then the concentration and deposition grids
             (and what the options add) are read back
  ensemble   perturbed scenarios stepped together, every scenario's grids read back
  adjoint    receptor concentrations of a release and the gradient of a weighted sum of them
  inversion  one iteration of the batched source inversion

The weather is homogeneous ("uniform", and "paper": Fig. 3b of the paper) or a seeded field
of the realistic kind: log wind plus mesoscale streamfunction modes, a weak vertical wind,
K_z from a similarity profile with a horizontally varying friction velocity, rain discs.

`exact` follows the same particles in 64 bits with torch alone: the counter-based generator
(Philox4x32-10) and the model's equations are written out below.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_0912_3223_gb300 import Sim, lpm
from paper_0912_3223_gb300.adjoint import receptor_concentrations
from paper_0912_3223_gb300.inversion import invert, observe

PLAIN = dict(form="plain", weather="realistic", particles=20_000, steps=2880, dt=30.0, nx=200,
             ny=200, nz=30, cells=400, layers=20, bin_every=120, rain=True, track=False,
             upload=False, eq3=False, dosage=0, langevin=False, species=1, gridded_kh=False,
             drift=False)
UNIFORM = dict(PLAIN, weather="uniform", particles=10_000, steps=360, dt=10.0, nx=2, ny=2, nz=2,
               cells=100, bin_every=360, rain=False, track=True)
ENSEMBLE = dict(form="ensemble", weather="realistic", scenarios=64, least=1e4, most=1e6,
                steps=720, dt=30.0, nx=200, ny=200, nz=30, cells=400, layers=1, modes=4, rain=True)
ADJOINT = dict(form="adjoint", weather="realistic", particles=1_000_000, steps=1080, dt=20.0,
               nx=200, ny=200, nz=30, cells=400, layers=20, side=8, every=18, trajectory=True,
               rain=True)
INVERSION = dict(ADJOINT, form="inversion", scenarios=16, particles=100_000)
BANDWIDTH = 200.0            # receptor kernel (m)
HALF_LIFE = 8 * 86400.0
CHAIN = (HALF_LIFE, 43200.0, 7200.0, 0.0)   # half-lives of a chain's species (s), the last stable


def listed():
    return [
        # the paper's own run (Fig. 3b: homogeneous weather, 6 h at 10 s): a run this small is
        # 2160 dependent steps and a few read-backs, so latency and launches count
        dict(UNIFORM, name="paper_2160x2160", weather="paper", particles=2160, steps=2160, nz=61,
             layers=15),
        # a quick look: uniform wind, ten thousand particles, one hour
        dict(UNIFORM, name="uniform_1e4x360"),
        # a day with a coarse particle budget, as while a run is being set up
        dict(PLAIN, name="day_2e4x2880"),
        # a six-hour forecast: the new weather comes from page-locked host memory in the same
        # call; a domain of odd sizes
        dict(PLAIN, name="forecast_1e6x720", particles=1_000_003, steps=720, nx=151, ny=133,
             nz=23, cells=301, layers=17, upload=True),
        # the headline run: ten million particles over a day
        dict(PLAIN, name="day_1e7x2880", particles=10_000_000),
        # a dose assessment: K_z from boundary-layer columns (Eq. 3), a time-integrated
        # dosage and a chain of three species
        dict(PLAIN, name="dose_eq3_chain_5e5x720", particles=500_000, steps=720, eq3=True,
             dosage=12, species=3),
        # near-source dispersion with velocity memory (Langevin) and a gridded K_h
        dict(PLAIN, name="langevin_kh_3e5x600", particles=300_000, steps=600, langevin=True,
             gridded_kh=True),
        # an ensemble of perturbed scenarios, and the small one of a sensitivity check
        dict(ENSEMBLE, name="ensemble_64x720"),
        dict(ENSEMBLE, name="ensemble_6x240", scenarios=6, least=500.0, most=3000.0, steps=240),
        # gradients of receptor concentrations: all states kept, and 64-step checkpoints
        dict(ADJOINT, name="adjoint_1e6x1080"),
        dict(ADJOINT, name="adjoint_ckpt_2e5x720", particles=200_000, steps=720,
             trajectory=False),
        # one iteration of the source inversion over all candidate sources
        dict(INVERSION, name="inversion_16x1e5"),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    grid = dict(nx=rng.randint(60, 220), ny=rng.randint(60, 220), nz=rng.randint(12, 40))
    kind = rng.choice(["uniform", "plain", "plain", "options", "ensemble", "adjoint", "inversion"])
    if kind == "uniform":
        steps = spread(90, 2200)
        return dict(UNIFORM, particles=spread(1000, 300_000), steps=steps, nz=rng.randint(2, 60),
                    cells=rng.randint(50, 150), bin_every=rng.choice([steps, 60, 97]))
    if kind in ("plain", "options"):
        c = {**PLAIN, **grid, "particles": spread(2000, 3_000_000), "steps": spread(120, 1800),
             "cells": rng.randint(150, 400), "layers": rng.randint(8, 20),
             "rain": rng.random() < 0.8, "bin_every": rng.choice([60, 77, 120, 240])}
        c["gridded_kh"] = rng.random() < 0.25
        if kind == "plain":
            c["drift"] = rng.random() < 0.25
            c["upload"] = rng.random() < 0.3
        else:
            c["eq3"] = rng.random() < 0.4
            c["langevin"] = not c["eq3"] and rng.random() < 0.5
            c["dosage"] = rng.choice([0, 4, 12, 25])
            c["species"] = rng.choice([1, 2, 3, 4])
        return c
    if kind == "ensemble":
        n = spread(2, 64)
        most = spread(2000, 300_000)
        return {**ENSEMBLE, **grid, "scenarios": n, "least": float(most // 10), "most": float(most),
                "steps": spread(60, 720), "cells": rng.randint(100, 400),
                "modes": rng.randint(0, 4), "rain": rng.random() < 0.8}
    c = {**ADJOINT, **grid, "particles": spread(2000, 500_000), "steps": spread(100, 1080),
         "side": rng.randint(3, 12), "every": rng.choice([6, 18, 25]),
         "trajectory": rng.random() < 0.6}
    if kind == "inversion":
        c.update(form="inversion", scenarios=spread(2, 16), particles=spread(1000, 60_000),
                 trajectory=True)
    return c


# ---- inputs ------------------------------------------------------------------------------
def _f32(v):
    """The value as single precision holds it (the model's parameters are read exactly)."""
    return float(np.float32(v))


def _weather(c, r):
    """Weather of a case on the GPU: uvwk [T][nz][ny][nx][4], kh, rain, bl, z_levels, spacing."""
    dev = "cuda"
    if c["weather"] != "realistic":
        nz, kz0 = c["nz"], 10.0
        top = 300.0 if c["weather"] == "paper" else 400.0
        z = np.linspace(0.0, top, nz)
        uvwk = torch.zeros(2, nz, 2, 2, 4, device=dev)
        u = 5.0 if c["weather"] == "paper" else _f32(r.uniform(3.0, 7.0))
        kz = np.full(nz, kz0)
        if c["weather"] == "paper":     # neutral log law through the source, Eq. 3 with Phi = 1
            ustar, hm = 0.4 * 5.0 / math.log(20.0 / 0.25), 120.0
            kz = np.where(z >= hm, 0.1, np.maximum(0.4 * ustar * z * (1 - z / hm) ** 2, 0.1))
        uvwk[..., 0] = u
        uvwk[..., 3] = torch.from_numpy(kz).to(dev)[None, :, None, None]
        return SimpleNamespace(uvwk=uvwk, kh=None, rain=None, bl=None, z=z, hours=2)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    T = max(2, int(math.ceil(c["steps"] * c["dt"] / 3600.0)) + 1)
    f8 = dict(device=dev, dtype=torch.float64)
    z = 3000.0 * (np.arange(nz) / (nz - 1)) ** 2
    zt = torch.from_numpy(z).to(dev)
    X, Y = torch.arange(nx, **f8)[None, :] * 250.0, torch.arange(ny, **f8)[:, None] * 250.0
    t = torch.arange(T, **f8)

    def waves(n, lo, hi, turn):
        out = []
        for _ in range(n):
            k, th = 2 * math.pi / math.exp(r.uniform(math.log(lo), math.log(hi))), r.uniform(0, 2 * math.pi)
            ph = r.uniform(0, 2 * math.pi) + t[:, None, None] * r.uniform(0.0, turn)
            out.append((math.cos(th), math.sin(th), torch.sin(k * (math.cos(th) * X + math.sin(th) * Y) + ph)))
        return out

    base = torch.where(zt > 0.1, torch.log(zt.clamp(min=0.1) / 0.1), zt * 0.0)     # u*/k = 1 m/s
    height = base / math.log(100.0 / 0.1)
    up, vp = torch.zeros(T, ny, nx, **f8), torch.zeros(T, ny, nx, **f8)
    for cs, sn, s in waves(16, 5e3, 5e4, 0.5 * math.pi):
        up -= 1.5 * math.sqrt(2.0 / 16) * sn * s
        vp += 1.5 * math.sqrt(2.0 / 16) * cs * s
    soft = [sum(w[2] for w in waves(4, 1e4, 4e4, 0.2)) / 2.0 for _ in range(4)]
    uvwk = torch.empty(T, nz, ny, nx, 4, device=dev)
    uvwk[..., 0] = base[None, :, None, None] + height[None, :, None, None] * up[:, None]
    uvwk[..., 1] = height[None, :, None, None] * vp[:, None]
    uvwk[..., 2] = (0.02 * torch.sin(math.pi * (zt / 3000.0)))[None, :, None, None] * soft[0][:, None]
    ustar = 0.4 * (1.0 + 0.2 * soft[1])
    prof = torch.where(zt < 1000.0, 0.4 * zt * (1 - zt / 1000.0) ** 2, zt * 0.0)
    uvwk[..., 3] = (prof[None, :, None, None] * ustar[:, None]).clamp(min=0.1)
    kh = bl = rain = None
    if c.get("gridded_kh"):
        kh = (100.0 * (1.0 + 0.3 * soft[2])).clamp(min=5.0)[:, None].expand(T, nz, ny, nx)
        kh = kh.to(torch.float32).contiguous()
    if c.get("eq3"):
        day = torch.sin(2 * math.pi * (t - 6) / 24.0)
        bl = torch.zeros(T, ny, nx, 4, device=dev)
        bl[..., 0] = ustar.clamp(0.1, 0.8)
        bl[..., 1] = torch.where(day > 0, -0.01 - 0.02 * day, 0.01 * (1.0 + day))[:, None, None] + 0.004 * soft[2]
        bl[..., 2] = ((1000.0 + 600.0 * day)[:, None, None] * (1.0 + 0.15 * soft[3])).clamp(200.0, 2500.0)
    if c["rain"]:
        lx = (nx - 1) * 250.0
        rain = torch.zeros(T, ny, nx, device=dev, dtype=torch.uint8)
        for _ in range(8):
            px, py, rad = r.uniform(-0.5, 1.0) * lx, r.uniform(0.0, 1.0) * (ny - 1) * 250.0, r.uniform(2e3, 5e3)
            at = (px + 6.9 * 3600.0 * t + 0.5 * lx) % (2.0 * lx) - 0.5 * lx
            rain |= ((X - at[:, None, None]) ** 2 + (Y - py) ** 2 <= rad * rad).to(torch.uint8)
    return SimpleNamespace(uvwk=uvwk, kh=kh, rain=rain, bl=bl, z=z, hours=T)


def _config(c, seed):
    """(configuration record, weather) of a case: the fields `Sim` reads."""
    r = random.Random(seed * 7919 + 17)
    w = _weather(c, r)
    n, steps = c.get("particles", 1), c["steps"]
    hours = int(math.ceil(steps * c["dt"] / 3600.0))

    def release(n):
        q = np.exp([r.gauss(0.0, 0.4) for _ in range(max(1, hours))])
        return SimpleNamespace(n_particles=n, q=q, q_dt=3600.0, first_step=0, last_step=steps)

    g = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], z_levels=w.z, n_met_t=w.hours, met_t0=0.0,
             met_dt=3600.0, cx=c["cells"], cy=c["cells"], cz=c["layers"], cz0=0.0, dt=c["dt"],
             n_steps=steps, seed=seed * 1000003 + 1, bin_every=c.get("bin_every", steps),
             reflect_ground=1, drift_correction=int(c.get("drift", False)), n_scenarios=1,
             uvwk=w.uvwk, kh=w.kh, rain=w.rain, scenarios=[], langevin=int(c.get("langevin", False)),
             t_lagr=100.0, kz_model=int(c.get("eq3", False)), kz_min=0.1, bl=w.bl, modes=None,
             mode_profile=None, chain_half_lives=None)
    if c.get("species", 1) > 1:
        g["chain_half_lives"] = np.array(CHAIN[: c["species"]])
    if c["weather"] == "realistic":
        lx, ly = (c["nx"] - 1) * 250.0, (c["ny"] - 1) * 250.0
        g.update(x0=0.0, y0=0.0, dx=250.0, dy=250.0, cx0=0.0, cy0=0.0, cdx=lx / c["cells"],
                 cdy=ly / c["cells"], cdz=50.0, src_x=_f32(0.1 * lx), src_y=_f32(ly * r.uniform(0.45, 0.55)),
                 src_z=50.0, half_life_s=HALF_LIFE, vd_dry=0.002, h_mix=1000.0,
                 wet_lambda=1e-4 if c["rain"] else 0.0,
                 kh_uniform=-1.0 if w.kh is not None else 100.0, reflect_top=1, z_top=3000.0,
                 lateral_exit=1)
    elif c["weather"] == "paper":
        g.update(x0=-1000.0, y0=-5000.0, dx=200000.0, dy=10000.0, cx0=-1000.0, cy0=-6000.0,
                 cdx=1200.0, cdy=120.0, cdz=20.0, src_x=0.0, src_y=0.0, src_z=20.0, half_life_s=0.0,
                 vd_dry=0.002, h_mix=120.0, wet_lambda=0.0, kh_uniform=100.0, reflect_top=1,
                 z_top=300.0, lateral_exit=0)
    else:
        g.update(x0=-1000.0, y0=-5000.0, dx=10000.0, dy=10000.0, cx0=-1000.0, cy0=-5000.0,
                 cdx=100.0, cdy=100.0, cdz=20.0, src_x=0.0, src_y=0.0, src_z=50.0, half_life_s=0.0,
                 vd_dry=0.0, h_mix=0.0, wet_lambda=0.0, kh_uniform=50.0, reflect_top=0, z_top=0.0,
                 lateral_exit=0)
    cfg = SimpleNamespace(**g)
    cfg.release = release(n)
    if c["form"] in ("ensemble", "inversion"):
        cfg.n_scenarios = c["scenarios"]
        if c.get("modes"):
            m = []
            for _ in range(c["modes"]):
                lam, th = math.exp(r.uniform(math.log(5e3), math.log(5e4))), r.uniform(0, 2 * math.pi)
                m.append([math.cos(th) / lam, math.sin(th) / lam, r.uniform(0, 0.25) / 3600.0,
                          -math.sin(th), math.cos(th)])
            cfg.modes = np.array(m, dtype=np.float32).astype(np.float64)
            prof = np.log(np.maximum(w.z, 0.1) / 0.1) / math.log(1000.0)
            cfg.mode_profile = prof.astype(np.float32).astype(np.float64)
        q = release(1).q
        for _ in range(c["scenarios"]):
            s = SimpleNamespace(wind_offset=None, mode_phase=None, mode_amp=None)
            s.src_x, s.src_y = _f32(lx * r.uniform(0.05, 0.25)), _f32(ly * r.uniform(0.25, 0.75))
            s.src_z = _f32(r.uniform(10.0, 300.0))
            if c["form"] == "ensemble":
                s.release = release(int(math.exp(r.uniform(math.log(c["least"]), math.log(c["most"])))))
                off, a = [], [r.gauss(0, 1.5), r.gauss(0, 1.5)]
                for _ in range(w.hours):
                    off.append(a)
                    a = [0.8 * v + 0.6 * r.gauss(0, 1.5) for v in a]
                s.wind_offset = np.array(off, dtype=np.float32)
                s.mode_phase = np.array([_f32(r.random()) for _ in range(c["modes"])])
                s.mode_amp = np.array([_f32(r.uniform(0.35, 1.05)) for _ in range(c["modes"])])
            else:
                s.release = release(c["particles"])
                s.release.q = q
            cfg.scenarios.append(s)
    cfg.n_particles = sum(s.release.n_particles for s in cfg.scenarios) or n
    return cfg, w


def _receptors(c, cfg):
    """side x side receptors at 2 m, downwind of the source and across the plume."""
    lx, ly = (c["nx"] - 1) * 250.0, (c["ny"] - 1) * 250.0
    xs = np.linspace(0.14 * lx, 0.5 * lx, c["side"])
    ys = np.linspace(0.4 * ly, 0.6 * ly, c["side"])
    X, Y = np.meshgrid(xs, ys, indexing="ij")
    rec = np.stack([X.ravel(), Y.ravel(), np.full(X.size, 2.0)], axis=1)
    return rec.astype(np.float32).astype(np.float64)


def _weights(c, seed):
    r = random.Random(seed + 5)
    return torch.tensor([[r.uniform(0.5, 1.5) for _ in range(c["side"] ** 2)]], dtype=torch.float64)


def prepare(case, seed):
    cfg, w = _config(case, seed)
    st = SimpleNamespace(case=case, cfg=cfg)
    if case["form"] == "inversion":
        r = random.Random(seed + 3)
        hidden = SimpleNamespace(**vars(cfg))
        hidden.n_scenarios, hidden.scenarios, hidden.seed = 1, [], cfg.seed + 1000
        hidden.src_x, hidden.src_y = cfg.src_x, cfg.src_y
        hidden.src_z = _f32(r.uniform(20.0, 150.0))
        hidden.release = cfg.scenarios[0].release
        hidden.n_particles = hidden.release.n_particles
        st.rec = _receptors(case, cfg)
        with Sim(hidden) as so:
            st.obs = observe(so, st.rec, BANDWIDTH, case["every"])
    st.sim = Sim(cfg)
    if case.get("upload"):
        st.host = [None if v is None else v.cpu().pin_memory() for v in (w.uvwk, w.kh, w.rain)]
    cfg.uvwk = cfg.kh = cfg.rain = cfg.bl = None         # the context has its own copy
    if case.get("dosage"):
        st.sim.set_dosage(case["dosage"])
    if case["form"] == "ensemble":
        shape = (case["scenarios"], case["cells"], case["cells"])
        st.conc = np.empty((shape[0], 1) + shape[1:])
        st.dep = np.empty((shape[0], 2) + shape[1:])
    if case["form"] == "adjoint":
        if not case["trajectory"]:
            lpm.lpm_set_adjoint_storage(st.sim.ctx, 0)
        st.rec, st.w = _receptors(case, cfg), _weights(case, seed)
        st.par = (torch.tensor([[cfg.src_x, cfg.src_y, cfg.src_z]], dtype=torch.float64),
                  torch.from_numpy(cfg.release.q)[None], torch.tensor(1.0, dtype=torch.float64),
                  torch.zeros(2, dtype=torch.float64))
    torch.cuda.synchronize()
    return st


def run(st):
    case, sim = st.case, st.sim
    if case["form"] == "inversion":
        res = invert(sim, st.rec, st.obs, n_iter=1, bandwidth=BANDWIDTH, every=case["every"])
        return {"sources": res.sources, "loss": res.loss, "grad": res.grad}
    if case["form"] == "adjoint":
        par = [p.clone().requires_grad_() for p in st.par]
        C = receptor_concentrations(sim, *par, st.rec, BANDWIDTH, case["every"])
        (C * st.w).sum().backward()
        return {"C": C.detach(), "sources": par[0].grad, "q": par[1].grad, "k_scale": par[2].grad,
                "bias": par[3].grad}
    if case.get("upload"):
        uvwk, kh, rain = st.host
        for t in range(st.cfg.n_met_t):
            lpm.lpm_set_met(sim.ctx, t, uvwk[t], None if kh is None else kh[t],
                            None if rain is None else rain[t])
    sim.reset()
    sim.step(case["steps"])
    if case["form"] == "ensemble":
        for s in range(case["scenarios"]):
            sim.concentration(s, out=st.conc[s])
            st.dep[s, 0], st.dep[s, 1] = sim.deposition(s)
        return {"conc": st.conc, "dep": st.dep}
    dry, wet = sim.deposition()
    out = {"conc": sim.concentration(), "dry": dry, "wet": wet}
    if case["track"]:
        out["xyz"], out["tag"] = sim.particles()
        out["budget"] = sim.budget()
    if case["dosage"]:
        out["dosage"] = sim.dosage()[0]
    if case["species"] > 1:
        out["species"] = [sim.species(j)[:3] for j in range(1, case["species"])]
    return out


def work(case):
    """Bytes: the weather that the run reads and the grids (or gradients) that it returns;
    flops: 399 32-bit operations a moving particle and step (two generator calls, the normals,
    16-corner interpolation of four fields, the move and the tests), twice that for a gradient's
    reverse step. A particle moves until the end of the run or until the wind carries it out."""
    hours = max(2, int(math.ceil(case["steps"] * case["dt"] / 3600.0)) + 1)
    life = case["steps"]
    if case["weather"] == "realistic":
        life = max(1.0, 0.9 * (case["nx"] - 1) * 250.0 / 6.9 / case["dt"])
    S = case["steps"]
    mean = S / 2 if life >= S else life - life * life / (2.0 * S)
    n = case.get("particles", 0)
    if case["form"] == "ensemble":
        a, b = case["least"], case["most"]
        n = case["scenarios"] * (a if a == b else (b - a) / math.log(b / a))
    if case["form"] == "inversion":
        n *= case["scenarios"]
    passes = {"plain": 1, "ensemble": 1, "adjoint": 3, "inversion": 4}[case["form"]]
    grids = 8.0 * case["cells"] ** 2 * (case["layers"] + 2) * case.get("species", 1)
    if case["form"] == "ensemble":
        grids *= case["scenarios"]
    if case["form"] in ("adjoint", "inversion"):
        grids = 8.0 * case.get("scenarios", 1) * (case["side"] ** 2 + 30)
    met = hours * case["nx"] * case["ny"] * (16.0 * case["nz"] + 1)
    return {"bytes": met + grids, "flops": 399.0 * n * mean * passes}


# ---- the same in 64 bits ------------------------------------------------------------------
def _philox(pid, step, stream, seed):
    """Philox4x32-10 (Salmon et al., SC'11): key = seed, counter = (pid low, high, step, stream);
    four int64 tensors holding 32-bit words."""
    m32 = 0xFFFFFFFF
    c = [pid & m32, pid >> 32, torch.full_like(pid, step), torch.full_like(pid, stream)]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _unit(w):
    return (2.0 * (w >> 9).double() + 1.0) * 2.0 ** -24


def _threshold(p):
    return min(4294967295, int(math.floor(p * 4294967296.0))) if p > 0 else 0


class _Exact:
    """The particles of every scenario of a configuration, in 64 bits."""

    def __init__(self, cfg, w, scen=None):
        self.cfg, self.w = cfg, w
        f8 = dict(device="cuda", dtype=torch.float64)
        self.z = torch.from_numpy(np.asarray(cfg.z_levels)).to(**f8)
        scen = scen or cfg.scenarios or [cfg]
        self.src = torch.tensor([[s.src_x, s.src_y, s.src_z] for s in scen], **f8)
        self.off = None
        if getattr(scen[0], "wind_offset", None) is not None:
            self.off = torch.tensor(np.stack([s.wind_offset for s in scen]), **f8)     # [S][T][2]
        self.modes = getattr(cfg, "modes", None)
        if self.modes is not None:
            self.ph = torch.tensor(np.stack([s.mode_phase for s in scen]), **f8)
            self.am = torch.tensor(np.stack([s.mode_amp for s in scen]), **f8)
            self.prof = torch.tensor(cfg.mode_profile, **f8)
        S = cfg.n_steps
        sp, sc, mass, per_q, hour = [], [], [], [], []
        for i, s in enumerate(scen):
            rel = s.release
            j = (torch.arange(rel.n_particles, device="cuda") * S) // rel.n_particles
            count = torch.bincount(j, minlength=S).double().clamp(min=1)
            h = (torch.arange(S, **f8) * cfg.dt / rel.q_dt).floor().long().clamp(max=len(rel.q) - 1)
            q = torch.tensor(np.asarray(rel.q), **f8)
            sp.append(j)
            sc.append(torch.full_like(j, i))
            per_q.append((cfg.dt / count)[j])
            hour.append(h[j])
            mass.append((q[h] * cfg.dt / count)[j])
        self.sp, self.sc, self.m0 = torch.cat(sp), torch.cat(sc), torch.cat(mass)
        self.per_q, self.hour = torch.cat(per_q), torch.cat(hour)
        order = torch.sort(self.sp, stable=True)
        self.order, self.upto = order.indices, torch.bincount(self.sp, minlength=S).cumsum(0).tolist()
        self.lam = math.log(2.0) / cfg.half_life_s if cfg.half_life_s > 0 else 0.0
        self.t_dry = _threshold(1 - math.exp(-cfg.vd_dry * cfg.dt / cfg.h_mix) if cfg.vd_dry > 0 else 0)
        self.t_wet = _threshold(1 - math.exp(-cfg.wet_lambda * cfg.dt)) if cfg.rain is not None else 0

    def axis(self, v, o, d, n):
        f = (v - o) / d
        i = f.detach().floor().clamp(0, n - 2)
        return i.long(), (f - i).clamp(0.0, 1.0)

    def level(self, z):
        k = (torch.searchsorted(self.z, z.detach().contiguous(), right=True) - 1).clamp(0, len(self.z) - 2)
        return k, ((z - self.z[k]) / (self.z[k + 1] - self.z[k])).clamp(0.0, 1.0)

    def slab(self, k):
        g = self.cfg
        ft = (k * g.dt - g.met_t0) / g.met_dt
        h = min(max(int(math.floor(ft)), 0), g.n_met_t - 2)
        return h, min(max(ft - h, 0.0), 1.0)

    def weather(self, k, x, y, z, sc):
        """(u, v, w, K_z, K_h, dK_z/dz) at the positions at the start of step k."""
        g = self.cfg
        h, f = self.slab(k)
        if getattr(self, "at", None) != k:
            blend = lambda a: a[h].double() * (1 - f) + a[h + 1].double() * f  # noqa: E731
            self.field = blend(g.uvwk).reshape(-1, 4)
            self.khf = None if g.kh is None else blend(g.kh).reshape(-1)
            self.blf = blend(g.bl).reshape(-1, 4) if g.kz_model else None
            self.at = k
        i, a = self.axis(x, g.x0, g.dx, g.nx)
        j, b = self.axis(y, g.y0, g.dy, g.ny)
        l, c = self.level(z)

        def bilinear(src, n):
            e = lambda v: v[:, None] if src.dim() == 2 else v  # noqa: E731
            lo = src[n] * (1 - e(a)) + src[n + 1] * e(a)
            hi = src[n + g.nx] * (1 - e(a)) + src[n + g.nx + 1] * e(a)
            return lo * (1 - e(b)) + hi * e(b)

        n = (l * g.ny + j) * g.nx + i
        lo, hi = bilinear(self.field, n), bilinear(self.field, n + g.nx * g.ny)
        r = lo * (1 - c[:, None]) + hi * c[:, None]
        u, v, w, kz = r.unbind(1)
        kh = torch.full_like(u, max(g.kh_uniform, 0.0))
        if self.khf is not None:
            kh = (bilinear(self.khf, n) * (1 - c) + bilinear(self.khf, n + g.nx * g.ny) * c).clamp(min=0.0)
        inside = (z >= self.z[0]) & (z <= self.z[-1])
        dkz = torch.where(inside, (hi[:, 3] - lo[:, 3]) / (self.z[l + 1] - self.z[l]), 0.0)
        kz = kz.clamp(min=0.0)
        if self.blf is not None:
            us, il, hz = bilinear(self.blf, j * g.nx + i).unbind(1)[:3]
            s, zeta = 1 - z / hz, z * il
            phi = torch.where(zeta >= 0, 1 + 5 * zeta, (1 - 16 * zeta.clamp(max=0.0)) ** -0.5)
            dphi = torch.where(zeta >= 0, torch.full_like(z, 5.0), 8 * (1 - 16 * zeta.clamp(max=0.0)) ** -1.5)
            on = (z > 0) & (z < hz) & (us > 0)
            kz = torch.where(on, 0.4 * us * z * s * s / phi, 0.0)
            dkz = torch.where(on, (0.4 * us * (s * s - 2 * z * s / hz) - kz * dphi * il) / phi, 0.0)
            dkz = torch.where(kz < g.kz_min, 0.0, dkz)
            kz = kz.clamp(min=g.kz_min)
        if self.off is not None:
            o = self.off[:, h] * (1 - f) + self.off[:, h + 1] * f
            u, v = u + o[sc, 0], v + o[sc, 1]
        if self.modes is not None and len(self.modes):
            p = self.prof[l] * (1 - c) + self.prof[l + 1] * c
            for m, (fx, fy, om, eu, ev) in enumerate(self.modes):
                s = self.am[sc, m] * torch.sin(2 * math.pi * (fx * x + fy * y + self.ph[sc, m] + om * k * g.dt))
                u, v = u + p * eu * s, v + p * ev * s
        return u, v, w, kz, kh, dkz

    def normals(self, pid, k):
        u = [_unit(w) for w in _philox(pid, k, 0, self.cfg.seed)]
        r0, r1 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
        return (r0 * torch.cos(2 * math.pi * u[1]), r0 * torch.sin(2 * math.pi * u[1]),
                r1 * torch.cos(2 * math.pi * u[3]))

    def move(self, k, pid, sc, sp, x, y, z, wv=None, scale=1.0, bias=(0.0, 0.0)):
        """The positions (and w') after step k."""
        g = self.cfg
        u, v, w, kz, kh, dkz = self.weather(k, x, y, z, sc)
        n0, n1, n2 = self.normals(pid, k)
        sh = torch.sqrt(2 * scale * kh * g.dt)
        xn, yn = x + (u + bias[0]) * g.dt + n0 * sh, y + (v + bias[1]) * g.dt + n1 * sh
        if g.langevin:
            s2, ds2 = kz / g.t_lagr, dkz / g.t_lagr
            low = s2 < 1e-6
            s2, ds2 = s2.clamp(min=1e-6), torch.where(low, 0.0, ds2)
            r = _philox(pid, k, 2, g.seed)
            start = torch.sqrt(s2) * torch.sqrt(-2 * torch.log(_unit(r[0]))) * torch.cos(2 * math.pi * _unit(r[1]))
            wv = torch.where(sp == k, start, wv)
            wv = wv - wv / g.t_lagr * g.dt + 0.5 * (1 + wv * wv / s2) * ds2 * g.dt + \
                torch.sqrt(2 * s2 * g.dt / g.t_lagr) * n2
            zn = z + (w + wv) * g.dt
        else:
            zn = z + w * g.dt + n2 * torch.sqrt(2 * scale * kz * g.dt)
            if g.drift_correction:
                zn = zn + dkz * g.dt
        for _ in range(4):
            flip = zn < 0
            zn, s = torch.where(flip, -zn, zn), torch.where(flip, -1.0, 1.0)
            if g.reflect_top:
                over = (zn > g.z_top) & ~flip
                zn, s = torch.where(over, 2 * g.z_top - zn, zn), torch.where(over, -s, s)
            wv = wv * s if g.langevin else wv
        zn = zn.clamp(min=0.0)
        return xn, yn, (zn.clamp(max=g.z_top) if g.reflect_top else zn), wv

    def fate(self, k, pid, x, y, z):
        """Status after step k: 0 moving, 2 dry, 3 wet, 4 out of the domain."""
        g = self.cfg
        st = torch.zeros_like(pid)
        if self.t_dry or self.t_wet:
            d = _philox(pid, k >> 1, 1, g.seed)[2 * (k & 1): 2 * (k & 1) + 2]
            if self.t_wet:
                i = ((x - g.x0) / g.dx + 0.5).floor().long().clamp(0, g.nx - 1)
                j = ((y - g.y0) / g.dy + 0.5).floor().long().clamp(0, g.ny - 1)
                h = min(max(int((k * g.dt - g.met_t0) // g.met_dt), 0), g.n_met_t - 1)
                st[(d[1] < self.t_wet) & (g.rain[h].reshape(-1)[j * g.nx + i] != 0)] = 3
            st[(d[0] < self.t_dry) & (z < g.h_mix)] = 2
        if g.lateral_exit:
            out = (x < g.x0) | (x > g.x0 + (g.nx - 1) * g.dx) | (y < g.y0) | (y > g.y0 + (g.ny - 1) * g.dy)
            st[out] = 4
        return st

    def follow(self, seen, states=None):
        """Every step; seen(k, pid, x, y, z, st) after each. With `states`, those of the moving
        particles before each step are kept there."""
        cuda = dict(device="cuda")
        pid = torch.empty(0, dtype=torch.int64, **cuda)
        X = torch.empty(4, 0, dtype=torch.float64, **cuda)
        for k in range(self.cfg.n_steps):
            new = self.order[(self.upto[k - 1] if k else 0): self.upto[k]]
            if len(new):
                src = self.src[self.sc[new]].T
                pid = torch.cat([pid, new])
                X = torch.cat([X, torch.cat([src, torch.zeros_like(src[:1])])], dim=1)
            if not len(pid):
                if states is not None:
                    states.append((pid, X[:3]))
                continue
            if states is not None:
                states.append((pid, X[:3]))
            x, y, z, wv = self.move(k, pid, self.sc[pid], self.sp[pid], *X)
            st = self.fate(k, pid, x, y, z)
            seen(k, pid, x, y, z, st)
            on = st == 0
            pid, X = pid[on], torch.stack([x, y, z, X[3] if wv is None else wv])[:, on]

    def cell(self, x, y, z=None):
        """Flat cell and whether it lies in the grid (without z: of the deposition grid)."""
        g = self.cfg
        i, j = ((x - g.cx0) / g.cdx).floor().long(), ((y - g.cy0) / g.cdy).floor().long()
        ok = (i >= 0) & (i < g.cx) & (j >= 0) & (j < g.cy)
        n = j * g.cx + i
        if z is not None:
            l = ((z - g.cz0) / g.cdz).floor().long()
            ok, n = ok & (l >= 0) & (l < g.cz), l * g.cy * g.cx + n
        return n, ok


def _amounts(half_lives, age):
    """Amounts of a chain's species per unit of the emitted parent after `age` (Bateman)."""
    lam = [math.log(2.0) / h if h > 0 else 0.0 for h in half_lives]
    out = []
    for j in range(len(lam)):
        s = 0.0
        for i in range(j + 1):
            den = math.prod(lam[k] - lam[i] for k in range(j + 1) if k != i)
            s = s + math.prod(lam[:j]) / den * torch.exp(-lam[i] * age)
        out.append(s)
    return out


def _exact_run(case, cfg, w):
    E = _Exact(cfg, w)
    S, f8 = cfg.n_scenarios, dict(device="cuda", dtype=torch.float64)
    chain = case.get("species", 1)
    plane, cube = cfg.cx * cfg.cy, cfg.cx * cfg.cy * cfg.cz
    conc, dep = torch.zeros(chain, S * cube, **f8), torch.zeros(chain, 2, S * plane, **f8)
    dose = torch.zeros(cube, **f8)
    N = len(E.sp)
    xyz, tag, lost = torch.empty(N, 3, **f8), E.sp.clone(), torch.zeros((), **f8)

    def seen(k, pid, x, y, z, st):
        nonlocal lost
        age = (k + 1 - E.sp[pid]).double() * cfg.dt
        m, sc = E.m0[pid] * torch.exp(-E.lam * age), E.sc[pid]
        dead = st != 0
        masses = [m] if chain == 1 else [E.m0[pid] * v for v in _amounts(CHAIN[:chain], age)]
        cell, ok = E.cell(x, y)
        for kind in (0, 1):
            hit = (st == 2 + kind) & ok
            for j, v in enumerate(masses):
                dep[j, kind].index_add_(0, (sc * plane + cell)[hit], v[hit])
        last = k == cfg.n_steps - 1
        if case.get("dosage") and (k + 1) % case["dosage"] == 0 or last:
            cell, ok = E.cell(x, y, z)
            ok = ok & ~dead
            if case.get("dosage") and (k + 1) % case["dosage"] == 0:
                dose.index_add_(0, cell[ok], m[ok])
            if last:
                for j, v in enumerate(masses):
                    conc[j].index_add_(0, (sc * cube + cell)[ok], v[ok])
        if case.get("track"):
            lost = lost + m[st == 4].sum()
            put = torch.ones_like(dead) if last else dead
            xyz[pid[put]] = torch.stack([x, y, z], dim=1)[put]
            tag[pid[put]] = (st[put] << 28) | E.sp[pid[put]]

    E.follow(seen)
    vol, area = cfg.cdx * cfg.cdy * cfg.cdz, cfg.cdx * cfg.cdy
    conc = (conc / vol).reshape(chain, S, cfg.cz, cfg.cy, cfg.cx)
    dep = (dep / area).reshape(chain, 2, S, cfg.cy, cfg.cx)
    if case["form"] == "ensemble":
        return {"conc": conc[0], "dep": dep[0].transpose(0, 1)}
    out = {"conc": conc[0, 0], "dry": dep[0, 0, 0], "wet": dep[0, 1, 0]}
    if case["track"]:
        out["xyz"], out["tag"] = xyz, tag
        moving = tag >> 28 == 0
        m = E.m0 * torch.exp(-E.lam * (cfg.n_steps - E.sp).double() * cfg.dt)
        ok = E.cell(xyz[:, 0], xyz[:, 1], xyz[:, 2])[1]
        b = [E.m0.sum(), m[moving & ok].sum(), m[moving & ~ok].sum()]
        for kind in (2, 3):
            b.append(E.m0[tag >> 28 == kind].sum())      # (no decay in the tracked cases)
        b += [lost, b[0] - b[1] - b[2] - b[3] - b[4] - lost, moving.double().sum()]
        out["budget"] = torch.stack(b)
    if case["dosage"]:
        out["dosage"] = (dose * case["dosage"] * cfg.dt / vol).reshape(cfg.cz, cfg.cy, cfg.cx)
    if chain > 1:
        out["species"] = [(conc[j, 0], dep[j, 0, 0], dep[j, 1, 0]) for j in range(1, chain)]
    return out


def _exact_adjoint(case, cfg, w, seed):
    """C by the forward, the gradient by autograd step by step backwards over the kept states
    (the events stay as they were)."""
    E = _Exact(cfg, w)
    rec = torch.from_numpy(_receptors(case, cfg)).cuda()
    wt = _weights(case, seed).cuda()[0]
    samples = cfg.n_steps // case["every"]
    C = torch.zeros(len(rec), dtype=torch.float64, device="cuda")
    norm, s2 = (2 * math.pi * BANDWIDTH ** 2) ** -1.5, BANDWIDTH ** 2

    def kernel(x, y, z, r):
        h2 = (x - r[0]) ** 2 + (y - r[1]) ** 2
        d1, d2 = h2 + (z - r[2]) ** 2, h2 + (z + r[2]) ** 2
        return norm * (torch.exp(-d1 / (2 * s2)) + torch.exp(-d2 / (2 * s2)))

    states, ended = [], []

    def seen(k, pid, x, y, z, st):
        on = st == 0
        ended.append(on)
        if (k + 1) % case["every"] == 0:
            m = E.m0[pid] * torch.exp(-E.lam * (k + 1 - E.sp[pid]).double() * cfg.dt)
            for i, r in enumerate(rec):
                C[i] += (m * kernel(x, y, z, r))[on].sum() / samples

    E.follow(seen, states)
    leaf = dict(dtype=torch.float64, device="cuda", requires_grad=True)
    scale, bias = torch.tensor(1.0, **leaf), torch.zeros(2, **leaf)
    mu = torch.zeros(3, len(E.sp), dtype=torch.float64, device="cuda")
    g_scale, g_bias = torch.zeros((), device="cuda").double(), torch.zeros(2, device="cuda").double()
    g_q = torch.zeros(len(cfg.release.q), dtype=torch.float64, device="cuda")
    n = len(ended)
    for k in range(cfg.n_steps - 1, -1, -1):
        pid, X = states.pop()
        if not len(pid):
            continue
        n -= 1
        X = X.detach().requires_grad_()
        x, y, z, _ = E.move(k, pid, E.sc[pid], E.sp[pid], *X, scale=scale, bias=bias)
        L = (mu[:, pid] * torch.stack([x, y, z])).sum()
        if (k + 1) % case["every"] == 0:
            unit = E.per_q[pid] * torch.exp(-E.lam * (k + 1 - E.sp[pid]).double() * cfg.dt) * ended[n]
            G = sum(wt[i] * kernel(x, y, z, r) for i, r in enumerate(rec)) * unit / samples
            g_q.index_add_(0, E.hour[pid], G.detach())
            L = L + (G * E.m0[pid] / E.per_q[pid]).sum()
        gX, gs, gb = torch.autograd.grad(L, (X, scale, bias))
        mu[:, pid] = gX
        g_scale, g_bias = g_scale + gs, g_bias + gb
    return {"C": C[None], "sources": mu.sum(1)[None], "q": g_q[None], "k_scale": g_scale, "bias": g_bias}


def exact(case, seed):
    if case["form"] == "inversion":     # three such sweeps over all candidates take longer
        return None
    with torch.no_grad() if case["form"] != "adjoint" else torch.enable_grad():
        cfg, w = _config(case, seed)
        return _exact_adjoint(case, cfg, w, seed) if case["form"] == "adjoint" else _exact_run(case, cfg, w)
