"""Launch-shape and sort-interval autotuner for the particle kernels.

Times complete runs (lpm_reset + lpm_step over the whole horizon, so the release ramp,
the exits and the end-of-run binning are all represented) for the library's own choice by
size and for every (threads per block, occupancy variant), and with ``autotune_with_sort``
also for several intervals of the re-ordering of the particles by weather cell (the steps
fused between two sorts), with CUDA events on the context stream, and keeps the fastest.
The library's choice is written ``None``, as in ``Sim``'s arguments. Results are cached per (GPU name, workload signature) in a JSON file
(``$LPM_AUTOTUNE_CACHE`` or ``~/.cache/lpm_gb300/autotune.json``). Every shape and sort
interval gives bit-identical results, so tuning never changes what is computed.
"""
from __future__ import annotations

import hashlib
import json
import os
from typing import Dict, Iterable, Optional, Tuple

from . import lpm

BLOCKS = (128, 256, 512)
OCCS = (0, 1, 2)
# shapes tried by default: the choice by size, which has shapes of its own (warps in pairs,
# several in one run), and every (block, tile factor 1, occupancy variant); the factor
# reaches no kernel
DEFAULT_SHAPES = [None] + [(b, 1, o) for b in BLOCKS for o in OCCS]


def cache_path() -> str:
    return os.environ.get("LPM_AUTOTUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "lpm_gb300",
                                       "autotune.json"))


def signature(cfg) -> str:
    """Workload signature: the shapes and switches that change the kernel's work."""
    parts = [cfg.nx, cfg.ny, cfg.nz, cfg.n_met_t, cfg.cx, cfg.cy, cfg.cz, cfg.n_steps,
             cfg.bin_every, cfg.n_particles, cfg.n_scenarios, cfg.kh is None,
             cfg.rain is None, cfg.vd_dry > 0, cfg.wet_lambda > 0, cfg.lateral_exit,
             cfg.reflect_top, cfg.drift_correction, round(cfg.dt, 6),
             getattr(cfg, "kz_model", 0), getattr(cfg, "chain_half_lives", None) is not None,
             0 if getattr(cfg, "modes", None) is None else len(cfg.modes)]
    return hashlib.sha1(repr(parts).encode()).hexdigest()[:16]


def _load() -> Dict:
    try:
        with open(cache_path()) as f:
            return json.load(f)
    except Exception:
        return {}


def _store(d: Dict) -> None:
    path = cache_path()
    try:
        os.makedirs(os.path.dirname(path), exist_ok=True)
        tmp = path + f".{os.getpid()}"
        with open(tmp, "w") as f:
            json.dump(d, f, indent=1, sort_keys=True)
        os.replace(tmp, path)
    except OSError:
        pass


Shape = Optional[Tuple[int, int, int]]


def _set_launch(sim, shape: Shape) -> None:
    if shape is None:
        lpm.lpm_set_auto(sim.ctx, launch=True, sort=False)
    else:
        lpm.lpm_set_launch(sim.ctx, *shape)


def _set_sort(sim, every: Optional[int]) -> None:
    if every is None:
        lpm.lpm_set_auto(sim.ctx, launch=False, sort=True)
    else:
        lpm.lpm_set_sort(sim.ctx, every)


def _label(shape: Shape) -> str:
    return "auto" if shape is None else "x".join(map(str, shape))


def time_shape(sim, shape: Shape, reps: int = 2) -> float:
    """Milliseconds of one complete run with the given launch shape (best of ``reps``)."""
    import torch
    _set_launch(sim, shape)
    stream = sim.stream
    best = float("inf")
    for _ in range(reps + 1):                # the first run builds graphs and warms up
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        sim.reset()
        sim.step(sim.cfg.n_steps - sim.k)
        e1.record(stream)
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def _fastest(sim, candidates, reps: int):
    """Times (label, shape, interval) candidates in turn (interval "keep": the context's);
    returns the fastest and the milliseconds of each."""
    results, chosen = {}, {}
    for label, shape, every in candidates:
        if every != "keep":
            _set_sort(sim, every)
        try:
            results[label] = time_shape(sim, shape, reps)
            chosen[label] = shape, every
        except lpm.LpmError as e:
            # shapes the context's options do not run with (dosage, Eq. 3 K_z, a decay chain,
            # the Langevin variant and perturbation modes need a tile factor of 1)
            if e.status != lpm.LPM_E_INVALID:
                raise
    if not results:
        raise RuntimeError("no launch shape runs with this context's options")
    return chosen[min(results, key=results.get)], results


def _shape(v) -> Shape:
    return None if v is None else tuple(int(x) for x in v)


# (the key names the candidates' generation: answers kept from before the choice by size was
# one of them are not served)
def _key(sim) -> str:
    import torch
    return f"{torch.cuda.get_device_name()}|{signature(sim.cfg)}|auto"


def autotune(sim, shapes: Optional[Iterable[Shape]] = None, use_cache: bool = True,
             reps: int = 2) -> Shape:
    """Picks and applies the fastest launch shape for ``sim`` (a ``Sim``); returns it (None:
    the library's choice by size)."""
    key = _key(sim)
    cache = _load() if use_cache else {}
    if key in cache:
        shape = _shape(cache[key]["shape"])
        _set_launch(sim, shape)
        return shape
    shapes = [_shape(v) for v in shapes] if shapes is not None else DEFAULT_SHAPES
    (shape, _), results = _fastest(sim, [(_label(v), v, "keep") for v in shapes], reps)
    _set_launch(sim, shape)
    sim.reset()
    if use_cache:
        cache = _load()
        cache[key] = {"shape": shape, "ms": results}
        _store(cache)
    return shape


# intervals tried by default: the choice by size, and none (0), 30, 60, 90 and 120 steps
SORT_INTERVALS = (None, 0, 30, 60, 90, 120)


def autotune_with_sort(sim, shapes: Optional[Iterable[Shape]] = None,
                       sort_intervals: Iterable[Optional[int]] = SORT_INTERVALS,
                       use_cache: bool = True,
                       reps: int = 2) -> Tuple[Shape, Optional[int], Dict[str, float]]:
    """Picks and applies the fastest (launch shape, sort interval) for ``sim``; returns the
    shape, the interval (None: the library's choice by size) and the measured milliseconds of
    every combination tried."""
    intervals = [None if e is None else int(e) for e in sort_intervals]
    key = f"{_key(sim)}|sort{intervals}"
    cache = _load() if use_cache else {}
    if key in cache:
        shape, every = _shape(cache[key]["shape"]), cache[key]["sort_every"]
        _set_launch(sim, shape)
        _set_sort(sim, every)
        return shape, every, cache[key]["ms"]
    shapes = [_shape(v) for v in shapes] if shapes is not None else DEFAULT_SHAPES
    (shape, every), results = _fastest(
        sim, [(f"{_label(v)}/sort{'auto' if e is None else e}", v, e)
              for e in intervals for v in shapes], reps)
    _set_launch(sim, shape)
    _set_sort(sim, every)
    sim.reset()
    if use_cache:
        cache = _load()
        cache[key] = {"shape": shape, "sort_every": every, "ms": results}
        _store(cache)
    return shape, every, results
