"""Autotuner for the row split of the iteration kernels.

The row kernels give each thread `rows_per_thread` rows (1, 2 or 4) of one
LP; the results do not depend on the choice, the speed does (more rows per
thread means more independent loads in flight per thread but fewer CTAs).  The
tuner times CUDA-graph replays of one representative LP of each size bucket (by
nonzeros) for every choice and keeps the fastest, cached in a JSON file keyed by
GPU name, kernel family, bucket and value precision.  The trials run the row
kernels also where the LP alone would run the resident kernel, which has no such
split: a batch that holds it may not fit there.  The best split depends on the
rows in flight (512 k nonzeros, FP32, 1 / 2 / 4 rows per thread: alone 17.2 / 18.9 /
28.1 us per iteration, 16 of them 197 / 150 / 139; 64 uneven LPs of 34 M together
799 / 599 / 504), so the trials of a batch run as many copies as it has nonzeros.
"""
from __future__ import annotations

import json
import os
import threading

from . import binding as B

CHOICES = (1, 2, 4)
CTA_CHOICES = (128, 256)
# nonzero-count buckets: [lo, hi)
BUCKETS = ((0, 1 << 17), (1 << 17, 1 << 19), (1 << 19, 1 << 21), (1 << 21, 1 << 62))
# iterations between evaluations in a trial: above the resident kernel's limit
ROW_N_EVAL = B.UC_RESIDENT_MAX_EVAL + 2
DEFAULT_CACHE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "tune_cache.json")
# a batch's trial holds at most so many nonzeros: with them the order of the choices is the
# large batches'
TRIAL_NNZ = 1 << 23


def copies_of(nnz: int, batch_nnz: int) -> int:
    """Copies of an LP that stand for a batch: a power of two, so that batches
    of about one size share their trials."""
    return 1 << (max(1, min(batch_nnz, TRIAL_NNZ) // max(nnz, 1)).bit_length() - 1)


def bucket_of(nnz: int) -> int:
    for i, (lo, hi) in enumerate(BUCKETS):
        if lo <= nnz < hi:
            return i
    return len(BUCKETS) - 1


class Tuner:
    def __init__(self, cache_path: str | None = DEFAULT_CACHE, trial_replays: int = 16):
        self.cache_path = cache_path
        self.trial_replays = trial_replays
        self._lock = threading.Lock()
        self.cache = {}
        if cache_path and os.path.exists(cache_path):
            try:
                with open(cache_path) as f:
                    self.cache = json.load(f)
            except (OSError, ValueError):
                self.cache = {}

    @staticmethod
    def _gpu_name() -> str:
        import torch
        return torch.cuda.get_device_name()

    def key(self, nnz: int, value_bits: int) -> str:
        return f"{self._gpu_name()}|rows|bucket{bucket_of(nnz)}|fp{value_bits}"

    def time_choice(self, ps, rpt: int, cta: int = 0, copies: int = 1) -> float:
        """Milliseconds per PDHG iteration of `copies` of `ps` with `rpt` rows per thread
        and `cta` threads per CTA (0: the library default) on the row kernels:
        graph replays of together at least 64 `trial_replays` iterations after
        one to warm up, timed on the device."""
        import torch
        n_eval = ROW_N_EVAL
        replays = 1 + max(1, -(-64 * self.trial_replays // n_eval))
        sess = B.Session([ps] * copies, tol=0.0, max_iter=n_eval * replays, n_eval=n_eval,
                         rows_per_thread=[rpt] * copies, cta_rows=cta)
        s = torch.cuda.current_stream()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        sess.reset(-1)
        sess.run(1)                      # warm-up: the reset's start-point evaluation and one replay
        e0.record(s)
        sess.run()                       # the remaining replays, steady state
        e1.record(s)
        torch.cuda.synchronize()
        sess.close()
        return e0.elapsed_time(e1) / (n_eval * (replays - 1))

    def choose(self, ps, value_bits: int, batch_nnz: int = 0) -> int:
        """Rows per thread for LPs of `ps`'s bucket, in a batch of `batch_nnz` nonzeros."""
        nnz = B.uc_presolved_dims(ps)[3]
        copies = copies_of(nnz, batch_nnz)
        k = self.key(nnz, value_bits) + (f"|x{copies}" if copies > 1 else "")
        with self._lock:
            if k in self.cache:
                return int(self.cache[k]["rows_per_thread"])
        kw = {"copies": copies} if copies > 1 else {}
        times = {r: self.time_choice(ps, r, **kw) for r in CHOICES}
        best = min(times, key=times.get)
        with self._lock:
            self.cache[k] = {"rows_per_thread": best, "ms_per_iter": times, "nnz_sample": nnz}
            if self.cache_path:
                tmp = self.cache_path + f".tmp{os.getpid()}"
                with open(tmp, "w") as f:
                    json.dump(self.cache, f, indent=1)
                os.replace(tmp, self.cache_path)
        return best

    def choose_pair(self, ps, value_bits: int) -> tuple[int, int]:
        """(threads per CTA, rows per thread) for a session holding `ps` alone."""
        nnz = B.uc_presolved_dims(ps)[3]
        k = "pair|" + self.key(nnz, value_bits)
        with self._lock:
            if k in self.cache:
                e = self.cache[k]
                return int(e["cta_rows"]), int(e["rows_per_thread"])
        # two rounds, interleaved, best of both: the choices differ by a few
        # percent, so each trial times a thousand steady-state iterations
        pairs = [(c, r) for c in CTA_CHOICES for r in CHOICES if r <= 2]
        times = {p: float("inf") for p in pairs}
        for _ in range(2):
            for c, r in pairs:
                times[(c, r)] = min(times[(c, r)], self.time_choice(ps, r, c))
        best = min(times, key=times.get)
        with self._lock:
            self.cache[k] = {"cta_rows": best[0], "rows_per_thread": best[1],
                             "ms_per_iter": {f"{c}x{r}": t for (c, r), t in times.items()}, "nnz_sample": nnz}
            if self.cache_path:
                tmp = self.cache_path + f".tmp{os.getpid()}"
                with open(tmp, "w") as f:
                    json.dump(self.cache, f, indent=1)
                os.replace(tmp, self.cache_path)
        return best
