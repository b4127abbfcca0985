"""Autotuner of the two-stage kernel's variant (the rows of a segment that a warp walks up).

Times each variant on the caller's own solver or batch and caches the winner
per (kind, precision, order, flux, size bucket) in a JSON file under the
user's cache directory. A timing is host wall-clock around a run of steps that
starts and ends with the object's stream drained (its status call waits for
it), so it measures that stream whatever stream the caller made current; the
run is long enough (at least ~2 ms of device work) that the launch and
synchronisation cost is small, and the best of three repeats is kept. The
variants run the same per-cell arithmetic (they agree to rounding; the tests
check it against the oracle and against each other), so the choice is a speed
one. Temporal blocking is not offered, on a measurement: the 1024^2 step with
its whole state resident in L2 between steps (what fusing steps would give) runs
only 5% faster than with L2 flushed before every step, while a second fused step
would recompute a halo of 60% more cells in an issue-bound kernel.
"""
from __future__ import annotations

import json
import math
import os
import time

# (2 is 4: both leave the choice to the library's rule)
VARIANTS = (0, 1, 3, 4, 5)


def _cache_path() -> str:
    base = os.environ.get("XDG_CACHE_HOME") or os.path.join(os.path.expanduser("~"), ".cache")
    return os.path.join(base, "dugks_gb300", "tune.json")


def _load() -> dict:
    try:
        with open(_cache_path()) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _store(d: dict):
    path = _cache_path()
    try:
        os.makedirs(os.path.dirname(path), exist_ok=True)
        tmp = path + f".{os.getpid()}"
        with open(tmp, "w") as f:
            json.dump(d, f, indent=1, sort_keys=True)
        os.replace(tmp, path)
    except OSError:
        pass


# bumped whenever a variant number changes its meaning (older cache entries are ignored)
TABLE = 3


def key(kind: str, params, cells: int) -> str:
    bucket = int(round(math.log2(max(cells, 1))))
    return f"t{TABLE}/{kind}/p{params.precision}/o{params.order}/f{params.flux}/c2^{bucket}"


def _time_steps(step_fn, sync_fn, steps: int) -> float:
    """Milliseconds per step of `steps` steps, stream drained on both sides."""
    sync_fn()
    t0 = time.perf_counter()
    step_fn(steps)
    sync_fn()
    return (time.perf_counter() - t0) * 1e3 / steps


def tune(obj, kind: str, cells: int, steps: int = 24, warmup: int = 8, use_cache: bool = True) -> int:
    """Pick the fastest variant for `obj` (a native.Solver or native.Batch), set it
    and return it. Unless the cache answers, the state advances by the warm-up and
    timed steps of every variant (a few hundred steps on small grids): tune a copy
    or restart from the initial field afterwards. The warm-up covers one full
    graph-replay chunk of a batch, so graph capture happens before the timed steps."""
    k = key(kind, obj.params, cells)
    cache = _load() if use_cache else {}
    if k in cache:
        obj.set_variant(int(cache[k]["variant"]))
        return int(cache[k]["variant"])
    times = {}
    for v in VARIANTS:
        obj.set_variant(v)
        obj.step(warmup)
        probe = _time_steps(obj.step, obj.status, steps)
        n = max(steps, int(math.ceil(2.0 / max(probe, 1e-4))))   # >= ~2 ms per timing
        times[v] = min(_time_steps(obj.step, obj.status, n) for _ in range(3))
    best = min(times, key=times.get)
    obj.set_variant(best)
    cache = _load()
    cache[k] = {"variant": best, "ms_per_step": times, "when": time.strftime("%Y-%m-%dT%H:%M:%S")}
    _store(cache)
    return best
