"""Autotuners of the stage's line kernel and of the batched launches.

Every variant computes identical results; only speed differs.  `autotune` times a few
js_step calls per variant with CUDA events on the solver's stream, selects the fastest and
caches the choice in a JSON file keyed by the kernels' sources, grid size, physics and immersed
body, so later solvers with the same key start tuned.  What a variant or a number of blocks
means is the kernels' business: a choice made for other sources is not applied.
"""
import functools
import hashlib
import json
import os

_HERE = os.path.dirname(os.path.abspath(__file__))
_CACHE = os.path.join(_HERE, "_build", "tuning.json")
# variants of the line kernel that differ (3 and 4 run variant 0's)
_VARIANTS = (0, 1, 2)


@functools.lru_cache(maxsize=None)
def _sources():
    """Short hash of the kernels' sources."""
    h = hashlib.sha1()
    d = os.path.join(_HERE, "csrc")
    for name in sorted(os.listdir(d)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(d, name), "rb") as f:
                h.update(name.encode() + b"\0" + f.read())
    return h.hexdigest()[:12]


def _key(solver):
    sp = solver._spec
    return "%s|%dx%d|visc=%d|av=%d|ib=%d" % (_sources(), sp["nx"], sp["ny"], int(sp["mu"] > 0), int(sp["nu"] > 0),
                                             int(getattr(solver, "has_ib", False)))


def _load():
    try:
        with open(_CACHE) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _save(cache):
    os.makedirs(os.path.dirname(_CACHE), exist_ok=True)
    tmp = _CACHE + ".tmp%d" % os.getpid()
    with open(tmp, "w") as f:
        json.dump(cache, f, indent=1, sort_keys=True)
    os.replace(tmp, _CACHE)


def cached_variant(solver):
    """The saved variant of this solver's key, or None."""
    v = _load().get(_key(solver), {}).get("variant")
    return v if v in _VARIANTS else None


def apply_cached(solver):
    v = cached_variant(solver)
    if v is not None:
        solver.set_tuning(v)
    return v


def autotune(solver, U, reps=3, use_cache=True):
    """Time the line kernel's variants that differ on state U (not modified) and select the fastest.
    Returns {variant: ms per step} ({} when the cache had the choice)."""
    import torch
    if use_cache and apply_cached(solver) is not None:
        return {}
    dt = 0.5 * solver.max_dt(U, 0.5)
    stream = torch.cuda.current_stream()
    times = {}
    work = U.clone()
    for v in _VARIANTS:
        solver.set_tuning(v)
        solver.step(work, dt, 1)  # warm-up (first launch sets kernel attributes)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record(stream)
        for _ in range(reps):
            solver.step(work, dt, 1)
        t1.record(stream)
        t1.synchronize()
        times[v] = t0.elapsed_time(t1) / reps
        work.copy_(U)
    # keep the default variant unless another is clearly faster
    best = min(times, key=times.get)
    if times[best] > 0.98 * times[0]:
        best = 0
    solver.set_tuning(best)
    cache = _load()
    cache[_key(solver)] = {"variant": best, "ms_per_step": times}
    _save(cache)
    return times


# ---------------------------------------------------------------------------------------
# batched path: blocks per SM and schedule of the forward's line kernels
# ---------------------------------------------------------------------------------------
def batch_key(problems):
    """The kernels' sources and the instance mix: grid sizes, physics and immersed bodies of all
    instances (order-free)."""
    items = sorted("%dx%d|visc=%d|av=%d|ib=%d" % (p.nx, p.ny, int(p.mu > 0), int(p.nu > 0), int(p.sdf is not None))
                   for p in problems)
    return "batch|%s|%d|%s" % (_sources(), len(items), hashlib.sha1("\n".join(items).encode()).hexdigest()[:16])


def cached_batch_choice(batch, problems):
    """The saved (blocks per SM, schedule) of this mix, or None; one out of the batch's range is not taken."""
    c = _load().get(batch_key(problems), {}).get("choice")
    _, most, _, nsched = batch.tuning()
    ok = isinstance(c, list) and len(c) == 2 and c[0] in range(most + 1) and c[1] in range(nsched)
    return tuple(c) if ok else None


def autotune_batch(batch, problems, states, steps=2, use_cache=True):
    """Time js_batch_step for every (blocks per SM, schedule) on copies of `states` (which are
    not advanced) and select the fastest; the choice is cached per instance mix.  Results are
    identical for every choice.  The batch's registered states are `states` afterwards.
    Returns {(blocks_per_sm, schedule): ms per step} ({} when the cache had the choice)."""
    import torch
    choice = cached_batch_choice(batch, problems) if use_cache else None
    if choice is not None:
        batch.set_tuning(*choice)
        batch.set_states(states)
        return {}
    _, most, _, nsched = batch.tuning()
    work = [U.clone() for U in states]
    batch.set_states(work)
    stream = torch.cuda.current_stream()
    times = {}
    for bps in range(1, most + 1):
        for sched in range(nsched):
            batch.set_tuning(bps, sched)
            for U, U0 in zip(work, states):
                U.copy_(U0)
            batch.step(0.5, 1)  # warm-up
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record(stream)
            batch.step(0.5, steps)
            t1.record(stream)
            t1.synchronize()
            times[(bps, sched)] = t0.elapsed_time(t1) / steps
    if batch.status() != 0:
        raise RuntimeError("batched tuning run failed")
    default = (most, 0)
    best = min(times, key=times.get)
    if times[best] > 0.98 * times[default]:
        best = default
    best = (best[0] % most, best[1])  # 0: the most that fit, whatever their number
    batch.set_tuning(*best)
    batch.set_states(states)
    cache = _load()
    cache[batch_key(problems)] = {"choice": list(best), "ms_per_step": {"%d,%d" % k: v for k, v in times.items()}}
    _save(cache)
    return times


def autotune_batch_reverse(batch, problems, states, dts, reps=2, use_cache=True):
    """Both settings of the reverse's launch form (js_batch_set_reverse_launch) run the same launches, so
    nothing is timed or cached: sets 0 and returns {}."""
    batch.set_reverse_launch(0)
    return {}
