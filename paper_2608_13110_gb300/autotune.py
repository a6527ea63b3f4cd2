"""Autotuner for the pass schedule.

The planner groups the paired steps of every absorbed row into windows of
address bits (the step-fusion depth of one HBM pass: up to 10 bits, i.e. up
to 9 steps per window and 16 at a row turn, whose four turn steps run as one
4x4 block). Which window sizes are fastest
depends on the width, the batch of bitstrings evaluated side by side, the GPU
and the circuit's gates: passes leave out entries that monomial gates make
exactly zero, and how many a pass can leave out depends on its window. So this
module times candidate schedules on the device, on circuits with that share of
monomial gates, and keeps the winner per (GPU, width, batch bucket, share of
monomial gates in thirds) in a JSON cache.

    from paper_2608_13110_gb300 import autotune
    opts = autotune.tune(h=24, nb=32)      # {"window_bits": .., "bottom_bits": .., "top_bits": ..}
    plan = autotune.tuned_plan(circuit, nb=32)
    opts = autotune.tune(h=24, nb=32, monomial=0.0)  # circuits of dense gates (Plan's extra)
"""
from __future__ import annotations

import json
import os
import threading

import numpy as np

from . import Plan

_LOCK = threading.Lock()
NARROW_MAX_WIDTH = 12  # whole boundary in one CTA: no windows to tune


def cache_path() -> str:
    return os.environ.get("TB_AUTOTUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "tbsweep", "autotune.json"))


def _load_cache() -> dict:
    try:
        with open(cache_path()) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _save_cache(c: dict) -> None:
    """Best effort: an unwritable cache only costs re-tuning later. Each
    process writes its own temporary file, then renames it into place."""
    p = cache_path()
    tmp = f"{p}.{os.getpid()}.tmp"
    try:
        os.makedirs(os.path.dirname(p) or ".", exist_ok=True)
        with open(tmp, "w") as f:
            json.dump(c, f, indent=1, sort_keys=True)
        os.replace(tmp, p)
    except OSError:
        try:
            os.remove(tmp)
        except OSError:
            pass


# Cliffords C_k = P_(k mod 4) . R_(k div 4) with one nonzero entry per row: R = I or S.
MONOMIAL = np.array([k // 4 in (0, 2) for k in range(24)])
UNIFORM = 1  # thirds of monomial gates among uniform random Cliffords (8 of 24)


def _thirds(monomial: float) -> int:
    return int(round(3.0 * min(1.0, max(0.0, monomial))))


def monomial_share(circ) -> float:
    """Share of a circuit's Cliffords that copy or flip a value (T gates keep that)."""
    return float(MONOMIAL[np.asarray(circ.cliff, np.int64)].mean())


def _bucket(nb: int) -> int:
    b = 1
    while b < nb:
        b *= 2
    return b


def candidate_options(h: int, n_rows: int = 8, limit: int = 8) -> list[dict]:
    """Feasible window choices for width h with distinct pass schedules,
    fewest passes first (ties: smallest largest pass)."""
    seen = {}
    d = 2 * h
    n = n_rows + 2
    for wb in (8, 9, 10):
        for bb in range(5, 11):
            for tt in range(5, 11):
                try:
                    p = Plan(n, d, window_bits=wb, bottom_bits=bb, top_bits=tt)
                except Exception:
                    continue
                sched = tuple(p.schedule)
                if sched in seen:
                    continue
                steps = [2 * m - 3 if s in ("top", "bot") else m for s, m, _ in sched]  # turn blocks count twice
                seen[sched] = ((len(sched), max(steps)), {"window_bits": wb, "bottom_bits": bb, "top_bits": tt})
    ranked = [v[1] for v in sorted(seen.values(), key=lambda kv: kv[0])]
    default = {"window_bits": 0, "bottom_bits": 0, "top_bits": 0}
    return [default] + ranked[: max(0, limit - 1)]


# Boundary entries the device keeps in flight per call by default (8 GiB of
# complex64): wider boundaries are evaluated one bitstring after another, so
# timing more of them measures nothing new.
BATCH_ENTRIES = 1 << 30


def measure(opts: dict, h: int, nb: int, n_rows: int = 8, reps: int = 3, seed: int = 1,
            monomial: float | None = None) -> float:
    """Milliseconds per batch of nb amplitudes of an (n_rows+2)-qubit circuit
    of width h under the given window options (median of reps): uniform random
    Cliffords, or a share ``monomial`` of monomial ones. A batch larger than the
    device evaluates at once is timed on the part it runs concurrently and
    scaled."""
    import torch
    import workloads as W
    run = max(1, min(nb, BATCH_ENTRIES >> h))
    scale = nb / run
    nb = run
    c = W.random_circuit(n_rows + 2, 2 * h, None, nb, seed)
    if monomial is not None:
        rng = np.random.default_rng(seed)
        pick = rng.random(c.cliff.shape) < monomial
        c.cliff = np.where(pick, rng.choice(np.flatnonzero(MONOMIAL), c.cliff.shape),
                           rng.choice(np.flatnonzero(~MONOMIAL), c.cliff.shape)).astype(np.uint8)
    plan = Plan.from_circuit(c, **opts)
    ws = plan.alloc_workspace(nb)
    plan.upload(ws)
    d_bits = torch.from_numpy(c.bits).cuda()
    out = torch.empty((nb, 2), dtype=torch.float64, device="cuda")
    plan.amplitudes_device(d_bits, ws, out)
    torch.cuda.synchronize()
    times = []
    for _ in range(reps):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        plan.amplitudes_device(d_bits, ws, out)
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    return float(np.median(times)) * scale


WIDE_LIMIT = 24  # candidates timed for boundaries of at least 2^WIDE_H entries
WIDE_H = 26


def tune(h: int, nb: int = 1, n_rows: int = 8, limit: int = 0, use_cache: bool = True,
         monomial: float | None = None) -> dict:
    """Fastest window options for width h with nb bitstrings side by side.
    monomial: share of the circuit's one-qubit gates that are monomial (None:
    uniform random Cliffords, a third of them).
    limit = 0 times 8 candidates, or 24 for widths >= 26: there the address
    span of a window changes the pass time (page and DRAM locality), which the
    planner's arithmetic cost model does not see."""
    if h <= NARROW_MAX_WIDTH:
        return {"window_bits": 0, "bottom_bits": 0, "top_bits": 0}
    if limit <= 0:
        limit = WIDE_LIMIT if h >= WIDE_H else 8
    import torch
    thirds = UNIFORM if monomial is None else _thirds(monomial)
    gates = {} if thirds == UNIFORM else {"monomial": thirds / 3.0}
    # entries without the share of monomial gates were timed on passes that visited every entry
    key = f"{torch.cuda.get_device_name()}|h={h}|nb={_bucket(nb)}|monomial={thirds}/3"
    with _LOCK:
        cache = _load_cache() if use_cache else {}
        if key in cache:
            return dict(cache[key]["opts"])
    results = []
    for opts in candidate_options(h, n_rows, limit):
        results.append((measure(opts, h, _bucket(nb), n_rows, **gates), opts))
    best_ms, best = min(results, key=lambda r: r[0])
    if use_cache:
        with _LOCK:
            cache = _load_cache()
            cache[key] = {"opts": best, "ms": best_ms, "tried": len(results)}
            _save_cache(cache)
    return dict(best)


def tuned_plan(circ, nb: int | None = None, **kw) -> Plan:
    """Plan for a circuit with autotuned window options."""
    h = (circ.d + 1) // 2
    kw.setdefault("monomial", monomial_share(circ))
    opts = tune(h, nb if nb is not None else max(1, circ.bits.shape[0]), **kw)
    return Plan.from_circuit(circ, **opts)
