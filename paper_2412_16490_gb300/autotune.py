"""Autotuner for the fused upper step.

Two knobs change how fast the step runs:

* the CTA tile, grasps per thread block (s lanes each): smaller tiles give
  more CTAs, so the grid spreads more evenly over the 152 SMs, at the price
  of partly filled warps (the tile never changes results).  Tile 0 leaves the
  choice to the library, which for ADMM at a fixed rho and a batch too small
  to fill the GPU takes the form with m lanes per QP; a requested tile runs
  one lane per QP;
* the lower-level schedule per upper step: ADMM with a fixed iteration
  count; ADMM to the 1e-5 residual up to a cap, warm-started from the
  previous upper step, its residuals checked every 10 or 25 iterations
  (fewer checks, up to 24 iterations past the target); or the exact solve
  (qp.solver = EXACT), warm-started from the previous step's working set.

`autotune` times every candidate on the workload over a full run and
returns the fastest acceptable one.  Two rules of acceptance:

* `residual=None`: the synthesis outcome, the median final energy within a
  tolerance of the reference schedule's (50 ADMM iterations per step);
* `residual=1e-5`: the QPs themselves, at least 99% of the grasps ending the
  run with every QP at or below 1e-5 (the ADMM residuals, or the exact
  solve's Frank-Wolfe gap, an upper bound on Q - Q*).

Every candidate's time, median energy and residual fraction are reported.
Results are cached per (template, wrench count, batch bucket, rule); a key
also names the candidate set, so that a file written when there were fewer
candidates is tuned again.
"""
from __future__ import annotations

import json
import os
import threading

import numpy as np

from . import QP_EXACT, State, bodex_step, qp_params, step_params

TILES = (0, 2, 4, 8)
SCHEDULES = (
    dict(mode="fixed", iters=20),
    dict(mode="fixed", iters=30),
    dict(mode="fixed", iters=50),
    dict(mode="converge", eps=1e-5, check=10, cap=200),
    dict(mode="converge", eps=1e-5, check=10, cap=1000),
    dict(mode="converge", eps=1e-5, check=25, cap=1000),
    dict(mode="exact", cap=64),
)
REFERENCE = dict(mode="fixed", iters=50)

CANDIDATES = "t0"  # in every key: changed with TILES and SCHEDULES

_cache: dict = {}
_lock = threading.Lock()


def schedule_qp(sched: dict, base: dict | None = None):
    """bodex_qp_params for a schedule."""
    b = dict(mu=0.5, beta=1.0, gamma=0.5, eps_reg=0.0)
    if base:
        b.update({k: base[k] for k in b if k in base})
    if sched["mode"] == "fixed":
        return qp_params(max_iter=sched["iters"], eps_abs=0.0, **b)
    if sched["mode"] == "exact":
        return qp_params(max_iter=sched["cap"], solver=QP_EXACT, **b)
    return qp_params(max_iter=sched["cap"], eps_abs=sched["eps"], check_every=sched["check"], **b)


def key_for(hand, s: int, B: int, residual=None) -> str:
    rule = "energy" if residual is None else f"res{residual:g}"
    return f"m{hand.m}-n{hand.n}-s{s}-B{1 << max(0, int(np.ceil(np.log2(max(B, 1)))))}-{rule}-{CANDIDATES}"


def autotune(hand, obj, x0, T, params: dict, steps: int = 200, energy_tol: float = 0.01, reps: int = 2,
             cache_path: str | None = None, tiles=TILES, schedules=SCHEDULES, reference=REFERENCE,
             residual: float | None = None, min_frac: float = 0.99) -> dict:
    """Pick (grasps_per_cta, lower-level schedule) for the fused step on this
    workload.  x0 [B, D] CUDA poses, T [s, 6].

    residual=None: a schedule is acceptable when the median energy after
    `steps` upper iterations is within `energy_tol` (relative) of the
    reference schedule's (50 ADMM iterations per step, as in the
    paper-scale runs).  residual=eps: when at least `min_frac` of the grasps
    end the run with every QP at a residual (ADMM) or Frank-Wolfe gap (exact
    solve) <= eps.  Returns the fastest acceptable pair with the whole
    table (the fastest of all when none is acceptable)."""
    import torch

    key = key_for(hand, int(T.shape[0]), int(x0.shape[0]), residual)
    with _lock:
        if key in _cache:
            return _cache[key]
        if cache_path and os.path.exists(cache_path):
            with open(cache_path) as f:
                disk = json.load(f)
            if key in disk:
                _cache[key] = disk[key]
                return disk[key]
    B, s = int(x0.shape[0]), int(T.shape[0])
    st = State(hand, B, s)
    E = torch.empty(B, dtype=torch.float32, device=x0.device)

    def run(sched, tile):
        sp = step_params(params, qp=schedule_qp(sched, params), grasps_per_cta=tile)
        times = []
        for r in range(reps + 1):
            st.set_pose(x0)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            bodex_step(hand, obj, st, T, steps, sp, E_last=E)
            b.record()
            torch.cuda.synchronize()
            if r:
                times.append(a.elapsed_time(b))
        lim = 1e-5 if residual is None else residual
        return float(np.median(times)), float(E.median().item()), float((st.residual() <= lim).float().mean().item())

    _, e_ref, _ = run(reference, 0)
    table = []
    for sched in schedules:
        for tile in tiles:
            ms, e_med, frac = run(sched, tile)
            good = e_med <= e_ref * (1.0 + energy_tol) if residual is None else frac >= min_frac
            table.append(dict(tile=tile, schedule=sched, ms=ms, median_E=e_med, frac_res_le_1e5=frac, ok=bool(good)))
    ok = [t for t in table if t["ok"]]
    best = min(ok or table, key=lambda t: t["ms"])
    out = dict(key=key, grasps_per_cta=best["tile"], schedule=best["schedule"], ms=best["ms"],
               median_E=best["median_E"], reference_median_E=e_ref, frac_res_le_1e5=best["frac_res_le_1e5"],
               steps=steps, energy_tol=energy_tol, residual=residual, min_frac=min_frac, table=table)
    with _lock:
        _cache[key] = out
        if cache_path:
            disk = {}
            if os.path.exists(cache_path):
                with open(cache_path) as f:
                    disk = json.load(f)
            disk[key] = out
            tmp = cache_path + f".tmp{os.getpid()}"
            with open(tmp, "w") as f:
                json.dump(disk, f, indent=1)
            os.replace(tmp, cache_path)
    return out


def tuned_params(tuned: dict, params: dict | None = None):
    """bodex_step_params for an autotune result."""
    return step_params(params, qp=schedule_qp(tuned["schedule"], params), grasps_per_cta=tuned["grasps_per_cta"])
