"""Sorted runs of every kernel family, whatever interval the library would pick for their size:
the sort, its key pass in the advance kernel, the sorted ranges in every default launch shape and
in fixed ones, mixed-scenario lanes, and the read-backs, saves and loads of sorted sets. Returns
their outputs; the checked-build test runs them once with each library and compares."""
import dataclasses

import numpy as np
import torch

import lpm_inputs as li

STEPS = 200


def cases() -> dict:
    """(configuration, Sim arguments, dosage interval) by name."""
    plain = li.make_cfg1(n_particles=4001, n_steps=STEPS, n_hours=4)
    chain = np.array([plain.half_life_s, 3600.0, 0.0])
    options = dataclasses.replace(plain, langevin=1, t_lagr=100.0, chain_half_lives=chain)
    ens = li.make_cfg2(n_scenarios=5, n_steps=STEPS, n_min=300, n_max=1500)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # the default shape above 8 warps an SM: everything leaves in the first 20 steps
    many = dataclasses.replace(li.make_cfg1(n_particles=8 * 32 * sms + 1, n_steps=STEPS, n_hours=4))
    many = dataclasses.replace(many, release=dataclasses.replace(many.release, last_step=20))
    sort, wide = {"sort_every": 30}, {"sort_every": 30, "launch": (512, 1, 2)}
    return {
        "plain": (plain, sort, 0), "plain_wide": (plain, wide, 0),
        "plain_many": (many, sort, 0),
        "eq3": (li.make_cfg1(n_particles=4001, n_steps=STEPS, n_hours=4, kz_eq3=True), sort, 0),
        "options": (options, sort, 8), "options_wide": (options, wide, 8),
        "ensemble": (ens, sort, 0), "ensemble_wide": (ens, wide, 0),
        "ensemble_options": (dataclasses.replace(ens, langevin=1, t_lagr=100.0), sort, 8),
    }


def run_case(cfg, kw, dosage) -> dict:
    """Steps in two pieces with a save and a load of the sorted set in between; every output."""
    from paper_0912_3223_gb300 import Sim, lpm
    out = {}
    with Sim(cfg, **kw) as sim:
        if dosage:
            sim.set_dosage(dosage)
        lpm.lpm_stats(sim.ctx)
        sim.step(STEPS // 2 + 3)
        out["launches"] = np.array(lpm.lpm_stats(sim.ctx)[0])
        blob = lpm.lpm_save(sim.ctx)
        out["blob"] = np.frombuffer(blob, np.uint8)
        lpm.lpm_load(sim.ctx, blob)
        sim.step(STEPS - STEPS // 2 - 3)
        out["xyz"], out["tag"] = sim.particles()
        if cfg.langevin:
            out["w"] = sim.velocity()
        for s in range(cfg.n_scenarios):
            out[f"conc{s}"], out[f"dep{s}"], out[f"ctr{s}"], _ = sim.fixed_state(s)
            out[f"budget{s}"] = sim.budget(s)
            if dosage:
                out[f"dose{s}"] = sim.dosage(s)[1]
            for j in range(1, 0 if cfg.chain_half_lives is None else 3):
                out[f"species{j}_{s}"], out[f"species{j}_dep{s}"] = sim.species(j, s)[3:]
    return out


def run_cases() -> dict:
    return {f"{name}_{k}": v for name, c in cases().items() for k, v in run_case(*c).items()}
