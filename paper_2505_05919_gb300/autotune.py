"""Autotuner of the batched kernel's tile shape and cells per thread.

A configuration is a tile of rows x 32-bit words (two cells per word) and the
block of threads that sweeps it; together they fix the cells each thread
updates per MC step, 2 rows words / threads.  The two dimensions are
searched as a product: four tiles (64 x 64, 32 x 32, 32 x 16, 16 x 16) with
256-thread blocks (32, 8, 4, 2 cells per thread), with 128-thread blocks
(64, 16, 8, 4) and with 512-thread blocks (16, 4, 2, 1).  Large tiles
amortise the recomputed one-cell ring and the staging; small ones give small
lattices enough tiles to fill the GPU; more cells per thread give each
thread more independent cells to interleave, fewer shorten the chain of one
tile's work (a small lattice's step is a chain of such tiles).

For a list of replica parameters the tuner builds a scratch batch with the
same lattice sizes (other seeds, so the caller's replicas are untouched),
times a short probe on every configuration with CUDA events, and returns
the fastest.  The automatic setting (-1) is not a configuration: where all
replicas are resident at once (up to about 1.2 million cells in at most 128
replicas) it runs without tiles and is faster than each of them (24 lattices of
64^2: 2.2 us per step against 8.9), and a configuration that is set switches
that off.  With ``automatic=True`` it is probed as well, and -1 is returned
where it wins.  Results are cached for the process by the mix of (L, q,
rng_words) and the probe length.  The state points (T, P) are not part of
the key: an arm update's accept or reject is a predicated select, so a
cell costs the same at any acceptance rate (the batched workload's sizes
timed on GB300 with its own (T, P) grid, all at 270 K / 0.1 MPa and all at
3000 K / 50 MPa: every configuration within 1 % of the same time, the same
one fastest).
"""
from __future__ import annotations

import copy

from . import _capi
from .batch import Batch, tile_configs

_cache: dict = {}


def signature(params_list) -> tuple:
    return tuple(sorted((p.L, p.q, p.rng_words) for p in params_list))


def cells_per_thread(config: int) -> int:
    """Cells one of the block's threads updates per MC step."""
    if config < 0:
        raise ValueError("the automatic setting has no tile of its own")
    rows, words, threads = tile_configs()[config]
    return 2 * rows * words // threads


def autotune(params_list, probe_sweeps: int = 20, warmup: int = 3, stream=None, automatic: bool = False):
    """Returns (best_config, {config: ms_per_step}) over the tile
    configurations and, with automatic, the automatic setting -1."""
    import torch
    key = (signature(params_list), probe_sweeps, automatic)
    if key in _cache:
        return _cache[key]
    scratch = []
    for p in params_list:
        q = copy.copy(p)
        q.seed = (p.seed * 2654435761 + 97) & 0xFFFFFFFFFFFFFFFF
        scratch.append(q)
    stream = stream if stream is not None else torch.cuda.Stream()
    timings = {}
    with Batch(scratch, stream=stream) as b:
        n = b.slots()
        for cfg in ([-1] if automatic else []) + list(range(len(tile_configs()))):
            b.set_tiles(cfg)
            b.sweep([warmup] * n)
            b.sync()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            b.sweep([probe_sweeps] * n)
            e1.record(stream)
            e1.synchronize()
            b.sync()
            timings[cfg] = e0.elapsed_time(e1) / probe_sweeps
    best = min(timings, key=timings.get)
    _cache[key] = (best, timings)
    return best, timings
