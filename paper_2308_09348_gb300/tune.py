"""Autotuner for the launch schedule (block size, tile size) of the kernels.

Candidates are timed on the caller's own problem with CUDA events after a
warm-up; the fastest is kept in a JSON cache keyed by the GPU name, the kernel
sources and a workload class string, so later runs of the same class skip the
search.  The histograms (integer sums) do not depend on the schedule; FP32
moments are summed in another grouping and may differ in their last digits.
"""
from __future__ import annotations

import ctypes
import functools
import hashlib
import json
import os
import threading
from collections import Counter

import torch

from . import binding as B
from . import build

_lock = threading.Lock()

# (block, tile); 0: left to the library, which chooses by kind of shot
BATCH_CANDIDATES = ((0, 0), (128, 512), (128, 1024), (128, 2048), (256, 512), (256, 1024),
                    (256, 2048), (256, 4096), (256, 8192))


def cache_path() -> str:
    base = os.environ.get("QSCATTER_CACHE_DIR") or os.path.join(
        os.path.expanduser("~"), ".cache", "libqscatter")
    return os.path.join(base, "autotune.json")


def _load() -> dict:
    try:
        with open(cache_path()) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def _store(db: dict) -> None:
    p = cache_path()
    os.makedirs(os.path.dirname(p), exist_ok=True)
    tmp = p + f".tmp{os.getpid()}"
    with open(tmp, "w") as f:
        json.dump(db, f, indent=1, sort_keys=True)
    os.replace(tmp, p)


def gpu_key() -> str:
    return torch.cuda.get_device_name(torch.cuda.current_device())


@functools.lru_cache(maxsize=1)
def sources_key() -> str:
    """Hash of the kernel sources (a schedule tuned for others is not reused)."""
    h = hashlib.sha1()
    for d in (build.CSRC, build.INCLUDE):
        for f in sorted(os.listdir(d)):
            with open(os.path.join(d, f), "rb") as src:
                h.update(f.encode() + b"\0" + src.read())
    return h.hexdigest()[:12]


def time_call(fn, reps: int = 3, warmup: int = 1) -> float:
    """Mean milliseconds of fn() on the current stream."""
    for _ in range(warmup):
        fn()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    a.record()
    for _ in range(reps):
        fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / reps


def tune(workload_class: str, candidates, make_runner, reps: int = 3, force: bool = False):
    """Return (best_candidate, {candidate: ms}).  make_runner(candidate) must
    return a zero-argument callable that performs one launch."""
    key = f"{gpu_key()}|{sources_key()}|{workload_class}"
    with _lock:
        db = _load()
        if not force and key in db:
            return tuple(db[key]["best"]), {tuple(json.loads(k)): v
                                            for k, v in db[key]["ms"].items()}
    times = {}
    for c in candidates:
        fn = make_runner(c)
        times[tuple(c)] = time_call(fn, reps=reps)
    best = min(times, key=times.get)
    with _lock:
        db = _load()
        db[key] = {"best": list(best), "ms": {json.dumps(list(k)): v for k, v in times.items()}}
        _store(db)
    return best, times


def batch_class(batch, n_total: int, weighted: bool = False) -> str:
    """Workload class of a ``binding.Batch``: what its time depends on."""
    raw = bytes(batch.d_lasers.cpu().numpy().tobytes())
    lasers = (B.qs_laser * batch.n_shots).from_buffer_copy(raw)
    assert ctypes.sizeof(lasers) == len(raw)
    mix = ",".join(f"{m}.{v}:{c}" for (m, v), c in
                   sorted(Counter((x.model, x.variant) for x in lasers).items()))
    b = batch.bins
    return (f"batch|shots={batch.n_shots}|mean={n_total // max(batch.n_shots, 1)}|"
            f"phase={batch.max_phase}|prec={batch.precision}|bins={b.n_bins}|"
            f"log={b.log_spaced}|smooth={b.smooth_sigma_bins:g}|map={b.n_tx}x{b.n_ty}|"
            f"aeff={b.n_aeff}|mix={mix}|sweep={int(batch.d_offsets is None)}|"
            f"weighted={int(weighted)}")
