"""Autotuner for the launch knobs of the persistent trace.

Knobs: threads per block (``block_threads``) and the level-buffer capacity
(``queue_capacity``, which sets how many rays one phase of the persistent schedule holds);
``chunk`` is still accepted in a search space, but the kernels take a warp's worth of rays at a
time whatever its value. Each candidate is timed with CUDA events on
a sample of the grid's sources (the cost of a trace is a sum over sources, so a sample ranks
the candidates like the whole set). A small sample separates the candidates that differ by
several percent but not the close ones, whose order can change with the number of sources in
flight, so the fastest few are timed again on a larger sample when the workload has more
sources than the first one. Candidates are timed with the outputs that the caller will ask for
(traces with and without a force are kernels of their own). The winner is cached in a JSON file
keyed by the grid shape, the number of sources, the base level, what selects the kernel (force,
cutoff) and the kernels' sources, so later runs of the same workload shape skip the search and
knobs found for other kernels are not used.
"""
from __future__ import annotations

import dataclasses
import hashlib
import itertools
import json
import os

import numpy as np
import torch

from . import art as A
from . import build

CACHE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_build", "tune_cache.json")

DEFAULT_SPACE = {
    "block_threads": [320, 640],
    "queue_capacity": [16 << 20, 64 << 20, 256 << 20],  # rays per deep-level buffer (4 B each)
}


def _kernel_version() -> str:
    """Digest of the trace kernels' sources."""
    h = hashlib.sha256()
    for name in ("art_kernels.cuh", "art_device.cuh"):
        with open(os.path.join(build.CSRC, name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:12]


def _key(shape, nsrc, params: A.Params, force: bool = True) -> str:
    return (f"{shape[0]}x{shape[1]}x{shape[2]}|src{nsrc}|l0{params.level0}|m{params.m_ray}"
            f"|cut{int(params.d_max > 0)}|force{int(force)}|{_kernel_version()}")


def _load_cache(path):
    try:
        with open(path) as f:
            return json.load(f)
    except Exception:
        return {}


def _time_knobs(g, params: A.Params, knobs: dict, repeats: int, stream, force: bool) -> float:
    """Best of ``repeats`` timed traces with these knobs (after one untimed trace, which also
    allocates); inf if the trace reports an error."""
    p = dataclasses.replace(params, schedule="persistent", **knobs)
    g.trace(p, force=force)
    best = float("inf")
    for _ in range(repeats):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        g.trace(p, force=force, stats=False)
        e1.record(stream)
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best if g.stats()["status"] == 0 else float("inf")


def tune(nH0: torch.Tensor, dx: float, pos, L, params: A.Params, sample: int = 16,
         space: dict | None = None, repeats: int = 2, cache_path: str | None = CACHE,
         nH: torch.Tensor | None = None, lo=(0.0, 0.0, 0.0), verbose: bool = False,
         refine_sample: int = 128, finalists: int = 3, force: bool = True) -> A.Params:
    """Returns ``params`` with the fastest knobs for this workload shape: every candidate
    timed on ``sample`` sources, then the ``finalists`` fastest on ``refine_sample`` sources
    (when the workload has more sources than the first sample). ``force``: whether the traces to
    come ask for the force."""
    pos = np.asarray(pos, dtype=np.float64).reshape(-1, 3)
    L = np.asarray(L, dtype=np.float64).reshape(-1)
    key = _key(tuple(nH0.shape), len(L), params, force)
    cache = _load_cache(cache_path) if cache_path else {}
    if key in cache:
        return dataclasses.replace(params, **cache[key]["knobs"])
    space = space or DEFAULT_SPACE
    rng = np.random.default_rng(0)
    idx = np.sort(rng.choice(len(L), size=min(sample, len(L)), replace=False))
    stream = torch.cuda.current_stream(nH0.device)
    g = A.Grid(nH0, dx, lo=lo, nH=nH, stream=stream)
    g.add_sources(pos[idx], L[idx])
    results = []
    names = list(space)
    for combo in itertools.product(*(space[n] for n in names)):
        knobs = dict(zip(names, combo))
        best = _time_knobs(g, params, knobs, repeats, stream, force)
        if best == float("inf"):
            continue
        results.append((best, knobs))
        if verbose:
            print(f"  {knobs}: {best:.3f} ms")
    g.close()
    if not results:
        raise RuntimeError("autotune: every candidate failed")
    results.sort(key=lambda r: r[0])
    nsample = len(idx)
    if finalists > 1 and len(L) > len(idx) and len(results) > 1:
        idx2 = np.sort(rng.choice(len(L), size=min(refine_sample, len(L)), replace=False))
        g = A.Grid(nH0, dx, lo=lo, nH=nH, stream=stream)
        g.add_sources(pos[idx2], L[idx2])
        refined = []
        for _, knobs in results[:finalists]:
            best = _time_knobs(g, params, knobs, repeats, stream, force)
            if best < float("inf"):
                refined.append((best, knobs))
            if verbose:
                print(f"  refined {knobs}: {best:.3f} ms")
        g.close()
        if refined:
            results = sorted(refined, key=lambda r: r[0])
            nsample = len(idx2)
    ms, knobs = results[0]
    if cache_path:
        cache = _load_cache(cache_path)
        cache[key] = {"knobs": knobs, "ms_sample": ms, "sample_sources": int(nsample),
                      "candidates": int(np.prod([len(v) for v in space.values()]))}
        os.makedirs(os.path.dirname(cache_path), exist_ok=True)
        tmp = cache_path + f".{os.getpid()}.tmp"
        with open(tmp, "w") as f:
            json.dump(cache, f, indent=1)
        os.replace(tmp, cache_path)
    return dataclasses.replace(params, **knobs)
