"""Autotuner for the launch choices of the TV library.

Two choices are measured on the running GPU and applied through the C ABI:
  * the largest batch of chains solved with warps per chain (latency-bound batches)
    rather than one thread per chain (throughput-bound batches). The library's own
    limits go with the chain length, the layout and the weights; one number for every
    batch, the crossover timed on uniform batches of 256- and 1024-node chains, takes
    their place only where it is the faster choice over batches of all kinds;
  * the warps per block of the batched 2D solver's persistent kernels, which run images
    with a side above 4096 pixels (others are on the splitting kernel).
Results are cached as JSON keyed by the GPU name and library version, in
``$TV_AUTOTUNE_CACHE`` or ``~/.cache/tv_gb300/autotune.json``.
"""
from __future__ import annotations

import json
import os

import numpy as np

from . import _lib, synth

CHOICES_WPB = (2, 4, 8)
BATCHES = (512, 1024, 2048, 4096, 8192)
LENGTHS = (256, 1024)
FORCE_COOP = 1 << 40
FORCE_THREAD = 1
# a GPU keeps the library's limits unless one crossover beats them by more than this
MARGIN = 0.02


def cache_path() -> str:
    return os.environ.get("TV_AUTOTUNE_CACHE",
                          os.path.join(os.path.expanduser("~"), ".cache", "tv_gb300",
                                       "autotune.json"))


def cache_key(device=0) -> str:
    import torch
    return f"{torch.cuda.get_device_name(device)}|tv{_lib.load().tv_version()}"


def _time_ms(fn, reps=5, warm=2):
    import torch
    for _ in range(warm):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return float(np.median(ts))


def choose_crossover(timings):
    """Largest batch at which the warp kernel is at least as fast as the thread
    kernel for every measured length; timings: {(B, n): (warp_ms, thread_ms)}."""
    best = 0
    for B in sorted({b for b, _ in timings}):
        rows = [timings[(b, n)] for (b, n) in timings if b == B]
        if all(w <= t for w, t in rows):
            best = B
        else:
            break
    return best


def keep_limits(own, crossover):
    """Whether the library's own limits stay: times of the same batches with them and with one
    crossover, compared by their geometric means."""
    ratio = np.exp(np.mean(np.log(np.asarray(own, float) / np.asarray(crossover, float))))
    return bool(ratio <= 1.0 / (1.0 - MARGIN))


def _mixed_batches(dev):
    """Batches of every kind around the library's limits, as calls."""
    import torch
    rng = np.random.default_rng(7)

    def rows(chains, n, edges):
        y = torch.from_numpy(np.tile(synth.chain_batch(50, n, seed0=n), (-(-chains // 50), 1))[:chains]).to(dev)
        w = torch.full_like(y, 0.15) if edges else None
        x = torch.empty_like(y)
        return lambda: _lib.chain_prox(y, w=w, lam=0.15, out=x)

    def columns(n, chains):
        y = torch.from_numpy(np.tile(synth.chain_batch(50, n, seed0=n), (chains // 50, 1)).T.copy()).to(dev)
        x = torch.empty_like(y)
        return lambda: _lib.chain_prox_columns(y, lam=0.15, out=x)

    def ragged(chains, longest):
        off = np.r_[0, np.cumsum(rng.integers(1, longest + 1, chains))]
        y = torch.from_numpy(np.resize(synth.chain_batch(50, 4096, seed0=3), off[-1])).to(dev)
        w, o = torch.full_like(y, 0.15), torch.from_numpy(off).to(dev)
        x = torch.empty_like(y)
        return lambda: _lib.chain_prox(y, w=w, offsets=o, max_len=longest, out=x)

    return [rows(512, 256, False), rows(4096, 1024, False), rows(16384, 512, False), rows(4096, 1023, True),
            rows(8192, 385, True), columns(512, 8000), ragged(6000, 2500), ragged(20000, 200)]


def measure(device=0):
    import torch
    dev = torch.device("cuda", device)
    timings = {}
    for n in LENGTHS:
        base = synth.chain_batch(256, n, seed0=1000)
        for B in BATCHES:
            y = torch.from_numpy(np.tile(base, (B // 256, 1))).to(dev)
            x = torch.empty_like(y)
            res = []
            for force in (FORCE_COOP, FORCE_THREAD):
                _lib.set_coop_max_chains(force)
                res.append(_time_ms(lambda: _lib.chain_prox(y, lam=0.15, out=x)))
            timings[(B, n)] = tuple(res)
    _lib.set_coop_max_chains(0)
    crossover = choose_crossover(timings)
    batches = _mixed_batches(dev)
    own = [_time_ms(fn) for fn in batches]
    _lib.set_coop_max_chains(max(crossover, 1))
    single = [_time_ms(fn) for fn in batches]
    _lib.set_coop_max_chains(0)
    # warps per block of the batched solver, on a small uneven batch of wide images
    sizes, lams = synth.uneven_image_sizes(6, seed=5, w_range=(4100, 4600), h_range=(32, 128))
    imgs = [torch.from_numpy(synth.shapes_image(h, w, seed=200 + i, n_shapes=40)[1]).to(dev)
            for i, (h, w) in enumerate(sizes)]
    wpb_ms = {}
    for wpb in CHOICES_WPB:
        _lib.set_batched_warps(wpb)
        wpb_ms[wpb] = _time_ms(lambda: _lib.tv2d_denoise_batched(imgs, lams, max_iters=100,
                                                                 tol=1e-4), reps=3, warm=1)
    best_wpb = min(wpb_ms, key=wpb_ms.get)
    return {"coop_max_chains": int(max(crossover, 1)), "batched_warps": int(best_wpb),
            "keep_limits": keep_limits(own, single),
            "mixed_ms": {"own_limits": own, "coop_max_chains": single},
            "chain_timings_ms": {f"{b}x{n}": list(v) for (b, n), v in timings.items()},
            "batched_warps_ms": {str(k): v for k, v in wpb_ms.items()}}


def apply(params):
    _lib.set_coop_max_chains(0 if params.get("keep_limits") else int(params["coop_max_chains"]))
    _lib.set_batched_warps(int(params["batched_warps"]))


def load_cache(path=None):
    path = path or cache_path()
    try:
        with open(path) as fh:
            return json.load(fh)
    except (OSError, ValueError):
        return {}


def save_cache(data, path=None):
    path = path or cache_path()
    os.makedirs(os.path.dirname(path), exist_ok=True)
    tmp = path + f".tmp{os.getpid()}"
    with open(tmp, "w") as fh:
        json.dump(data, fh, indent=1, sort_keys=True)
    os.replace(tmp, path)


def autotune(device=0, force=False, path=None):
    """Tuned parameters for this GPU (measured once, then read from the cache), applied."""
    key = cache_key(device)
    data = load_cache(path)
    if force or key not in data:
        data[key] = measure(device)
        save_cache(data, path)
    apply(data[key])
    return data[key]
