"""Autotuner for the block capacity C and the edge-kernel organisation.

The paper ties C to the thread-block size and picks it by hand (Section 5,
Table 3: blocks of 256, 512 and 1024 tasks).  Here C (tasks per schedule
block) and the kernel organisation (pipeline stages, threads per CUDA block;
stages 0: one CUDA block per kernel block) are separate knobs, chosen by
measurement in the regime the batch runs in, where the state and task data
do not fit in the L2:

1. screening: a seeded sample of the graphs is partitioned by the library for
   every candidate C and merged into one schedule; one forward step plus one
   adjoint step is timed for every (stages, threads) candidate with CUDA
   events, `reps` times, with the L2 flushed (a write of twice its size)
   before every repetition;
2. confirmation: the `confirm` fastest screening rows are timed again the same
   way on the whole set of graphs, and the fastest of those wins.

What is timed, and so what is tuned, are the step kernels: single steps, and
runs and gradients of batches that do not fit the chip.  Where a batch does fit
(Schedule.grad_sizes(D) is not zero) its runs and gradients take neither stages
nor threads from here, and C only sets the order that the parts are cut from.

Results are cached in a JSON file keyed by a hash of the graphs and the
candidate lists, so a rerun skips the search.
"""
from __future__ import annotations

import hashlib
import json
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np

from . import Schedule

DEFAULT_CS = (256, 512, 1024)
DEFAULT_KERNELS = ((3, 192), (2, 192), (3, 128), (3, 256), (2, 256), (4, 256), (0, 160), (0, 256))
CACHE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_build", "autotune.json")


def partition_many(graphs, C: int, threads: int = 0, workers: int | None = None):
    """Partition (n, src, dst) graphs concurrently (the library call releases the GIL)."""
    workers = workers or max(1, os.cpu_count() or 1)
    per_call = 1 if len(graphs) >= workers else threads

    def one(g):
        n, s, d = g
        return Schedule.partition(s, d, n, C, threads=per_call)

    with ThreadPoolExecutor(max_workers=workers) as ex:
        return list(ex.map(one, graphs))


def _key(graphs, Cs, kernels, D, extra):
    h = hashlib.sha256()
    for n, s, d in graphs:
        h.update(np.int64(n).tobytes())
        h.update(np.ascontiguousarray(s).tobytes())
        h.update(np.ascontiguousarray(d).tobytes())
    h.update(repr((tuple(Cs), tuple(kernels), D, extra)).encode())
    return h.hexdigest()[:24]


class _Flush:
    """Evicts the L2 between timed repetitions (a write of twice its size)."""

    def __init__(self, torch):
        l2 = torch.cuda.get_device_properties(torch.cuda.current_device()).L2_cache_size
        self.buf = torch.empty(max(2 * l2, 64 << 20) // 4, dtype=torch.float32, device="cuda")

    def __call__(self):
        self.buf.zero_()


def _time_configs(torch, B, D, configs, reps, tau, flush):
    """Mean ms of one forward + one adjoint step of schedule B for every (stages, threads)."""
    x = torch.randn(D, B.n, device="cuda")
    w = torch.rand(B.m, device="cuda") + 0.5
    xl = torch.empty(B.layout_floats(D), device="cuda")
    wl = torch.empty(B.weights_floats(), device="cuda")
    lam = torch.empty_like(xl)
    gw = torch.zeros_like(wl)
    B.layout_in(x, xl)
    B.layout_in(x, lam)
    B.weights_in(w, wl)
    out = []
    for stages, threads in configs:
        B.set_pipeline(stages)
        B.set_threads(threads)

        def step():
            B.step(D, xl, xl, wl, None, tau)
            B.adjoint_step(D, xl, wl, lam, gw, tau)

        step()
        torch.cuda.synchronize()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(reps)]
        for a, b in ev:
            flush()
            a.record()
            step()
            b.record()
        torch.cuda.synchronize()
        out.append(float(np.mean([a.elapsed_time(b) for a, b in ev])))
    return out


def tune(graphs, D: int = 5, Cs=DEFAULT_CS, kernels=DEFAULT_KERNELS, sample: int = 32,
         reps: int = 20, seed: int = 0, cache: str | None = CACHE, tau: float = 1e-3,
         confirm: int = 3, partitions: dict | None = None):
    """Best {C, stages, threads} for flux steps on these graphs (list of (n, src, dst)).

    `partitions`, if given, receives the full-set schedules partitioned during
    the confirmation ({C: [Schedule per graph]}), so the caller can reuse them."""
    import torch

    key = _key(graphs, Cs, kernels, D, ("v2", sample, reps, seed, confirm))
    if cache and os.path.exists(cache):
        try:
            with open(cache) as fh:
                hit = json.load(fh).get(key)
            if hit:
                return hit
        except (OSError, ValueError):
            pass
    rng = np.random.default_rng(seed)
    idx = np.sort(rng.choice(len(graphs), size=min(sample, len(graphs)), replace=False))
    sub = [graphs[i] for i in idx]
    flush = _Flush(torch)
    table = []
    for C in Cs:
        B = Schedule.batch(partition_many(sub, C))
        for (stages, threads), ms in zip(kernels, _time_configs(torch, B, D, kernels, reps, tau, flush)):
            table.append(dict(C=C, stages=stages, threads=threads, ms=ms, ns_per_task=1e6 * ms / B.m))
        B.close()
    top = sorted(table, key=lambda r: r["ns_per_task"])[: max(1, confirm)]
    confirmed = []
    for C in sorted({r["C"] for r in top}):
        parts = partition_many(graphs, C)
        if partitions is not None:
            partitions[C] = parts
        B = Schedule.batch(parts)
        cfgs = [(r["stages"], r["threads"]) for r in top if r["C"] == C]
        for (stages, threads), ms in zip(cfgs, _time_configs(torch, B, D, cfgs, reps, tau, flush)):
            confirmed.append(dict(C=C, stages=stages, threads=threads, ms=ms, ns_per_task=1e6 * ms / B.m))
        B.close()
    best = min(confirmed, key=lambda r: r["ms"])
    out = dict(C=best["C"], stages=best["stages"], threads=best["threads"], table=table,
               confirmed=confirmed, sample=[int(i) for i in idx], reps=reps, l2="flushed")
    if cache:
        os.makedirs(os.path.dirname(cache), exist_ok=True)
        try:
            with open(cache) as fh:
                allc = json.load(fh)
        except (OSError, ValueError):
            allc = {}
        allc[key] = out
        with open(cache, "w") as fh:
            json.dump(allc, fh)
    return out
