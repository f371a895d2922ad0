"""Autotuner of the multigrid launch shape of a grid.

The tunables change the preconditioner of the pressure solve, never the
converged answer (every candidate solves to the same poisson_rtol):

  mg_coarse_cells -- levels of at most this many cells are handled together
                     by one coarse V-cycle launch (fewer, longer launches
                     against more, shorter ones; 0: the library's rule; no
                     effect on 2D grids whose whole solve is one launch);
  mg_pre, mg_post -- red-black sweeps before and after the coarse correction
                     (cheaper V-cycles against fewer CG iterations);
  sweep_tile      -- 3D mixed precision, tuned second with the best shape
                     fixed: the column tile and cells per thread of the
                     TMA-staged finest-level sweep (more warps per SM against
                     less per-plane control per cell; smaller against larger
                     staged halos);
  inner_tol       -- optional (tune_inner), mixed precision only, tuned
                     second with the best shape fixed: the residual reduction
                     of each float32 inner solve between float64 refinements
                     (fewer refinements against fewer inner iterations). On
                     the uneven 2D batch it gave no gain beyond run-to-run
                     spread, so it is off by default.

Each candidate gets a fresh context on the same parameters, runs `warm`
steps, then `steps` timed steps (pf_step synchronises, so the host clock
brackets device work; candidates that are one and the same on a 2D grid solved
in one launch are timed once); the fastest candidate wins, except that the library's
defaults are kept unless a candidate beats them by more than MARGIN (a few
timed steps do not resolve smaller differences). Results are cached per
signature in memory and, given a path, in a JSON file, so a batch of many
instances tunes each grid size once.
"""
from __future__ import annotations

import json
import os
import time

CANDIDATES = tuple(
    [{"mg_coarse_cells": c, "mg_pre": v, "mg_post": v} for v in (1, 2) for c in (1024, 0, 16384)]
    + [{"mg_coarse_cells": c, "mg_pre": v, "mg_post": v} for v in (3, 4, 6) for c in (0, 16384)]
    + [{"mg_coarse_cells": 0, "mg_pre": v, "mg_post": v} for v in (8, 10)])

DEFAULT_SHAPE = {"mg_coarse_cells": 0, "mg_pre": 1, "mg_post": 1}   # the library's defaults
MARGIN = 0.01                            # relative gain needed to leave a default

INNER_TOLS = (1e-6, 1e-5, 1e-4, 1e-3)   # the first is the library's default
SWEEP_TILES = (0, 1, 2, 3, 4)           # the first is the library's default

# Part of every cache key: raised whenever the candidates or what the library makes
# of them change, so that a stored choice is not used for something else (1:
# mg_coarse_cells 4096 was the default, 2: 0, the library's rule)
SETTINGS_VERSION = 2

_cache: dict = {}


def signature(p: dict, tune_inner: bool = False) -> str:
    """What the best launch shape depends on: the version of the settings, the grid, precision, model,
    force, density ratio, walls, execution mode, the solve's tolerances (a
    tight poisson_rtol favours stronger V-cycles; a preset inner_tol is part of
    the problem) and whether the inner tolerance was tuned as well."""
    n = tuple(int(v) for v in p["n"])
    ratio = round(float(p["rho_in"]) / float(p["rho_out"]), 6)
    return json.dumps([f"v{SETTINGS_VERSION}", int(p["dim"]), n, str(p.get("precision")), str(p.get("model")),
                       str(p.get("force")), ratio, int(p.get("wall_y", 0) or 0),
                       int(p.get("use_graph", 0) or 0), float(p.get("poisson_rtol", 0.0) or 0.0),
                       float(p.get("inner_tol", 0.0) or 0.0), bool(tune_inner)])


def _time_candidate(pf, p: dict, cand: dict, steps: int, warm: int) -> float:
    sim = pf.Simulation(dict(p, **cand))
    try:
        sim.step(warm)
        t0 = time.perf_counter()
        sim.step(steps)
        return (time.perf_counter() - t0) / steps
    finally:
        sim.close()


def _one_launch(pf, p: dict) -> bool:
    """Whether the 2D grid's solves run in one launch, where mg_coarse_cells has no
    effect."""
    sim = pf.Simulation(dict(p))
    try:
        sim.step(1)
        return pf.pf_profile_read(sim.ctx).get("solve2d_cluster", (0, 0.0))[0] > 0
    finally:
        sim.close()


def tune(p: dict, candidates=CANDIDATES, steps: int = 2, warm: int = 1,
         cache_path: str | None = None, tune_inner: bool = False) -> dict:
    """Best candidate for the parameters p: {"choice": {...}, "ms_per_step":
    {candidate: ms}, "cached": bool}."""
    import paper_2205_05835_gb300 as pf

    key = signature(p, tune_inner)
    if key not in _cache and cache_path and os.path.exists(cache_path):
        with open(cache_path) as f:
            _cache.update(json.load(f))
    if key in _cache:
        return dict(_cache[key], cached=True)
    times, same, one_launch = {}, {}, None
    for c in candidates:
        k = json.dumps(c, sort_keys=True)
        first = same.setdefault(json.dumps(dict(c, mg_coarse_cells=0), sort_keys=True), k)
        if first != k and int(p["dim"]) == 2:
            # differs in mg_coarse_cells alone
            if one_launch is None:
                one_launch = _one_launch(pf, p)
            if one_launch:
                times[k] = times[first]
                continue
        times[k] = 1e3 * _time_candidate(pf, p, c, steps, warm)
    # of equal ones the library's own rule
    best = min(times, key=lambda k: (times[k], json.loads(k).get("mg_coarse_cells", 0) != 0))
    dkey = json.dumps(DEFAULT_SHAPE, sort_keys=True)
    if dkey in times and times[dkey] <= times[best] * (1.0 + MARGIN):
        best = dkey
    choice = json.loads(best)
    if int(p["dim"]) == 3 and p.get("precision") == "mixed" and "sweep_tile" not in p:
        base_ms = times[best]
        best_tile_ms, choice_t = base_ms, choice
        for tile in SWEEP_TILES[1:]:
            c = dict(choice, sweep_tile=tile)
            ms = 1e3 * _time_candidate(pf, p, c, steps, warm)
            times[json.dumps(c, sort_keys=True)] = ms
            if ms < base_ms * (1.0 - MARGIN) and ms < best_tile_ms:
                best_tile_ms, choice_t = ms, c
        choice = choice_t
    if tune_inner and p.get("precision") == "mixed" and not p.get("inner_tol"):
        base_ms = times[json.dumps(choice, sort_keys=True)]
        for tol in INNER_TOLS[1:]:
            c = dict(choice, inner_tol=tol)
            ms = 1e3 * _time_candidate(pf, p, c, steps, warm)
            times[json.dumps(c, sort_keys=True)] = ms
            if ms < base_ms:
                base_ms, choice = ms, c
    res = {"choice": choice, "ms_per_step": times}
    _cache[key] = res
    if cache_path:
        with open(cache_path, "w") as f:
            json.dump(_cache, f)
    return dict(res, cached=False)


def apply(p: dict, res: dict) -> dict:
    """p with the tuned launch shape."""
    return dict(p, **res["choice"])
