"""Autotuner for batched sweeps: picks the launch shape of a batch by timing.

The knobs (ccmc_batch_config) are the most threads per CTA of the resident
launches (64 to 512), the CTAs per SM the lattices share out among them, the
largest lattice kept in shared memory (the shared-memory path; the rest take the
per-phase L2/HBM path; a batch that was never configured keeps what ccmc_sweep
would), and the most threads that share one packed word of a lattice (1, 2 or 4:
the pairs each thread evaluates, 16, 8 or 4).  None of them changes results -- the random
streams are keyed by (seed, phase, site) -- so the tuner may pick freely.

A probe batch of synthetic lattices with the same shapes is swept for a few
sweeps under the library's own plan (a batch that was never configured) and under
every candidate, twice each (the faster probe counts).  The times are cached in a
JSON file (paper_2301_11735_gb300/_build/autotune.json) keyed by the GPU name, the
batch's shape signature and a digest of the library's sources: times taken with
other kernels say nothing about these.
"""
from __future__ import annotations

import hashlib
import json
import os
import time

_HERE = os.path.dirname(os.path.abspath(__file__))
_CACHE = os.path.join(_HERE, "_build", "autotune.json")

# (threads per CTA, largest resident lattice in sites, CTAs per SM, most
# threads a word): the argument order of Batch.config
DEFAULT = (256, 1 << 17, 2, 4)
CANDIDATES = [
    (threads, resident, ctas, tpw)
    for threads in (128, 256)
    for resident in (1 << 12, 1 << 14, 1 << 17)
    for ctas in (2, 4)
    for tpw in (1, 4)
] + [(64, 1 << 17, 2, 4), (256, 1 << 17, 2, 2), (512, 1 << 17, 1, 2), (512, 1 << 17, 1, 4),
     (512, 1 << 17, 1, 1)]


def _gpu_name() -> str:
    try:
        import torch

        return torch.cuda.get_device_name()
    except Exception:
        return "cuda"


def signature(shapes) -> str:
    counts = {}
    for s in shapes:
        counts[tuple(s)] = counts.get(tuple(s), 0) + 1
    key = ",".join(f"{a}x{b}:{n}" for (a, b), n in sorted(counts.items()))
    return hashlib.sha1(key.encode()).hexdigest()[:16]


def _sources() -> str:
    """Digest of the sources that the library is built from."""
    h = hashlib.sha1()
    for d in (os.path.join(_HERE, "csrc"), os.path.join(os.path.dirname(_HERE), "include")):
        for name in sorted(os.listdir(d) if os.path.isdir(d) else ()):  # a copy without sources
            with open(os.path.join(d, name), "rb") as f:
                h.update(name.encode() + b"\0" + f.read())
    return h.hexdigest()[:16]


def _load():
    try:
        with open(_CACHE) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _store(cache):
    os.makedirs(os.path.dirname(_CACHE), exist_ok=True)
    tmp = _CACHE + f".tmp{os.getpid()}"
    with open(tmp, "w") as f:
        json.dump(cache, f, indent=1, sort_keys=True)
    os.replace(tmp, _CACHE)


def _probe(shapes, probe_sweeps, params):
    """Seconds of probe_sweeps sweeps of a batch of `shapes`, by launch shape (None:
    the library's own plan)."""
    import paper_2301_11735_gb300 as cc

    lats = []
    for i, (Lx, Ly) in enumerate(shapes):
        lat = cc.Lattice(Lx, Ly)
        lat.init_constrained(7919 + i, 0.1, 0.3)
        lats.append(lat)
    timings = {}
    with cc.Batch(lats) as b:
        for cand in [None] + CANDIDATES:
            if cand is not None:
                try:
                    b.config(*cand)
                except cc.CcmcError:
                    continue
            b.sweep(2, *params)  # warm-up
            b.sync()
            best = float("inf")
            for _ in range(2):  # the faster of two probes: one noisy probe picked a slower shape
                t0 = time.perf_counter()
                b.sweep(probe_sweeps, *params)
                b.sync()
                best = min(best, time.perf_counter() - t0)
            timings[cand] = best
    for lat in lats:
        lat.close()
    return timings


def measured(shapes, probe_sweeps: int = 20, params=(1.0, 0.0, 1.0, 1.0),
             use_cache: bool = True) -> dict:
    """What the probes of a batch of `shapes` say: "config", the fastest candidate;
    "plan", whether a batch that is not configured at all is at least as fast (one with
    lattices of more than about 360 x 360 is, which no candidate holds in shared memory:
    20 of 512 x 512 take 15 us a sweep, not 40); "timings_ms"."""
    key = f"{_gpu_name()}|{signature(shapes)}|{len(DEFAULT)}|{_sources()}"
    cache = _load() if use_cache else {}
    if key not in cache:
        timings = _probe(shapes, probe_sweeps, params)
        configs = {c: t for c, t in timings.items() if c is not None}
        best = min(configs, key=configs.get) if configs else DEFAULT
        entry = {"config": list(best),
                 "plan": None in timings and timings[None] <= configs.get(best, float("inf")),
                 "timings_ms": {str(c and list(c)): 1e3 * t for c, t in timings.items()}}
        if not configs:
            return entry
        cache[key] = entry
        _store(cache)
    return cache[key]


def tune(shapes, probe_sweeps: int = 20, params=(1.0, 0.0, 1.0, 1.0), use_cache: bool = True):
    """Best (threads, resident_max_sites, ctas_per_sm, max_threads_per_word) for a batch
    of `shapes`, of the candidates."""
    return tuple(measured(shapes, probe_sweeps, params, use_cache)["config"])
