"""Tile-shape autotuner for the fused step kernel and the batch kernel.

The shape is (threads per CTA, rows per CTA), of which the library takes the rows (the grid's width decides its threads):
they trade pipeline fill (a segment of h rows runs h + 7 row iterations, the first and last few with stages idle) for
parallelism (one CTA per strip x segment).  The library's own choice is always measured too and stays unless
another is faster by more than MARGIN; the other heights are a fixed list and those that put a whole wave of one or two
CTAs per SM on the device (one row less can add a nearly empty wave).  Each runs about a millisecond of steps timed with
CUDA events on the simulation's stream, and the winner is cached per (device, grid class, storage and forms, kernel source)
in a JSON file next to the library (git-ignored).
"""
from __future__ import annotations

import hashlib
import json
import os
import threading

HERE = os.path.dirname(os.path.abspath(__file__))
CACHE = os.path.join(HERE, "_autotune_cache.json")
AUTO = "auto"                    # set_tile's value for the library's own rows; 0 in results
MARGIN = 0.01                    # by which another height has to be faster
THREADS = (128, 64, 256)         # accepted by set_tile, without effect: each height is measured once
ROWS = (1, 2, 4, 8, 12, 15, 16, 20, 24, 32, 48, 64, 96, 128)
MAX_CTAS_PER_SM = 2
STRIP = 2 * 122 + 6              # columns of the widest strip and its halo
_lock = threading.Lock()


def _kernel_hash():
    h = hashlib.sha256()
    for f in ("lbm_device.cuh", "lbm_march.cuh", "lbm_rows.cuh", "lbm_api.cu"):   # (the last: the library's own heights)
        with open(os.path.join(HERE, "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def _device_name():
    import torch
    return torch.cuda.get_device_name(torch.cuda.current_device()).replace(" ", "_")


def grid_class(nx, ny):
    """Grids of similar shape share a tuned tile: round sizes up to powers of two."""
    def up(v):
        p = 32
        while p < v:
            p *= 2
        return p
    return "%dx%d" % (up(nx), up(ny))


def _load():
    if os.path.exists(CACHE):
        try:
            with open(CACHE) as f:
                return json.load(f)
        except (OSError, ValueError):
            return {}
    return {}


def _store(cache):
    tmp = CACHE + ".tmp%d" % os.getpid()
    with open(tmp, "w") as f:
        json.dump(cache, f, indent=1, sort_keys=True)
    os.replace(tmp, CACHE)


TUNER_VERSION = "own-choice-1"    # entries measured over another candidate set are not reused


def _key(kind, nx, ny, params):
    forms = "s%df%d" % (int(getattr(params, "s_form", 0)), int(getattr(params, "f_form", 0)))
    return "|".join((kind, _device_name(), _kernel_hash(), grid_class(nx, ny), "st%d" % int(params.storage), forms, TUNER_VERSION))


def _time(fn, reps, stream):
    import torch
    fn()                                            # warm-up (graph capture, attributes)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    for _ in range(reps):
        fn()
    b.record(stream)
    b.synchronize()
    return a.elapsed_time(b) / reps


def _sm_count():
    import torch
    return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count


def balanced_rows(nx, ny, span, sms, max_per_sm=MAX_CTAS_PER_SM):
    """For each k = 1..max_per_sm, the shortest height h whose CTA count strips x ceil(ny / h)
    is at most k x sms (strips of at most span - 6 columns)."""
    strips = -(-nx // (span - 6))
    out = []
    for k in range(1, max_per_sm + 1):
        segs = (k * sms) // strips
        if segs < 1:
            continue
        h = -(-ny // segs)
        if h not in out:
            out.append(h)
    return out


def sim_candidates(nx, ny, sms):
    """(threads, rows) pairs for an nx x ny simulation on a device with `sms` SMs."""
    rows = sorted(set(ROWS) | set(balanced_rows(nx, ny, STRIP, sms)))
    return [(t, r) for t in THREADS for r in rows]


def _fastest(times):
    """(threads, rows, ms) of the fastest of `times`, with rows 0 for the library's own choice, which is measured last and
    has the benefit of MARGIN."""
    best = min(times, key=lambda e: e[2])
    own = times[-1]
    if own[1] == AUTO and own[2] <= best[2] * (1.0 + MARGIN):
        best = own
    return (best[0], 0 if best[1] == AUTO else best[1], best[2])


def _reps_for(fn, stream, target_ms=1.0, lo=6, hi=400):
    """Repetitions that make a timed run last about target_ms."""
    one = _time(fn, 2, stream)
    return max(lo, min(hi, int(target_ms / max(one, 1e-4))))


def tune_sim(sim, reps=None, candidates=None, use_cache=True):
    """Measure tile candidates on `sim` (its state advances; re-initialise it afterwards) and
    set the fastest.  Returns (threads, rows, ms per step), rows 0 for the library's own choice (which a new
    simulation has, and set_tile with 0 leaves).  `candidates`: those pairs alone.  `reps` None: about a millisecond of
    steps per candidate."""
    import torch
    key = _key("sim", sim.nx, sim.ny, sim.params)
    with _lock:
        cache = _load() if use_cache else {}
    if key in cache:
        t, r, ms = cache[key]
        sim.set_tile(t, r or AUTO)
        return t, r, ms
    stream = torch.cuda.current_stream()
    sim.set_stream(stream)
    times, seen = [], set()
    for t, r in candidates or sim_candidates(sim.nx, sim.ny, _sm_count()) + [(THREADS[0], AUTO)]:
        h = r if r == AUTO else min(r, sim.ny)      # taller segments are the whole grid
        if h in seen:
            continue
        seen.add(h)
        sim.set_tile(t, r)
        n = reps if reps else _reps_for(lambda: sim.step(1), stream)
        times.append((t, r, _time(lambda: sim.step(1), n, stream)))
    best = _fastest(times)
    sim.set_tile(best[0], best[1] or AUTO)
    if use_cache:
        with _lock:
            cache = _load()
            cache[key] = list(best)
            _store(cache)
    return best


BATCH_THREADS = (128,)
BATCH_ROWS = (16, 24, 32, 48, 64, 96, 128, AUTO)


def tune_batch(batch, reps=3, candidates=None):
    """Measure (threads, rows) of the batch kernel on the current membership (members advance) and set the fastest.
    Returns (threads, rows, ms per step), rows as in tune_sim."""
    import torch
    stream = torch.cuda.current_stream()
    times = []
    for t, r in candidates or [(t, r) for t in BATCH_THREADS for r in BATCH_ROWS]:
        batch.set_tile(t, r)
        times.append((t, r, _time(lambda: batch.step(2), reps, stream) / 2))      # per step
    best = _fastest(times)
    batch.set_tile(best[0], best[1] or AUTO)
    return best
