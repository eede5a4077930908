"""Continuous-batching search server on one GPU.

Systems (determinants, coefficients, E0, integrals) are registered once and
stay resident on the device.  Requests name a system and (C, N) and are
admitted in arrival order as soon as a slot is free and their device-memory
footprint fits the budget; admitted searches run concurrently, each on its
own CUDA stream from its own worker thread, so requests that arrive while
others are on the GPU join them as slots and memory free up.  Each search
caps its constraint batches to its memory share, so a result does not depend
on what else is running (the batch size does not change any output).
"""
from __future__ import annotations

import collections
import math
import threading
import time
from concurrent.futures import Future

import numpy as np

from . import search as _search, FP64

__all__ = ["Server", "footprint"]


def footprint(norb: int, ndets: int, C: int, N: int, batch_pairs: int, *, na: int | None = None,
              nb: int | None = None, alphas: int | None = None, group: int | None = None) -> int:
    """Upper estimate of one search's device bytes beyond its resident inputs (N = 0: of
    ASCI-PT2's), from the sizes of its allocations.  ``alphas`` is the number of distinct
    alpha strings of psi and ``group`` the most determinants of one of them (both C by
    default).  Without the electron counts half of the orbitals are taken, the counts of
    most pairs, and a batch is taken to fill its cap."""
    def pairs2(k):
        return k * (k - 1) // 2

    known = na is not None and nb is not None
    na, nb = (na, nb) if known else (norb // 2, norb // 2)
    C = min(C, ndets)
    alphas = min(C, C if alphas is None else alphas)
    group = min(C, C if group is None else group)
    # operations on an alpha string, and pairs of a determinant: o = 0, an alpha single
    singles, doubles = na * (norb - na), pairs2(na) * pairs2(norb - na)
    beta = nb * (norb - nb)
    npd0, npd1 = beta + pairs2(nb) * pairs2(norb - nb), 1 + beta
    P = C * (npd0 + singles * npd1 + doubles)
    items = alphas * (1 + singles + doubles)
    # pairs of a batch: the cap, or one target alpha string's, which no cap divides
    cap = batch_pairs or 1 << 31
    b = max(min(P, cap) if known else cap, min(P, group * npd0 + C * npd1))
    it = min(items, b)                                # items of a batch
    strings = min(it, math.comb(norb, na))            # and their target alpha strings
    runs = b // npd1 + b // 64 + (b // npd0 if npd0 else 0)
    tiles = b // 256 + 2
    cells = b // 400 + 1
    appended = N + max(1024 * 152 * 16, min(b, 1 << 29))  # candidate pool
    psi = (24 + 1 + 8 + 64) * ndets + 8192            # keys, sort, selection, hash table
    core = (8 * norb + 120) * C
    tables = 28 * norb ** 4 + 64 * norb ** 3 + (13 << 20)
    plan = 29 * items + 60 * min(items, math.comb(norb, na))
    staging = 20 * (b + b // 2 + (1 << 16))
    pool = 32 * appended
    lists = 40 * it + 60 * strings + 8 * runs + 32 * tiles + 16 * cells + 16 * ndets + b // 64
    # records beyond their bucket's slots: the list, and one as long as it takes with its
    # sort; then the oversized buckets' records gathered (on chip with their value
    # buffers, or sorted)
    big = b if b > 1024 else 0
    spilled = 20 * max(1 << 20, b // 32) + 37 * big + 41 * big
    # value buffers of a launch: 48 lists and 512 values a tile, or room for every record
    # of a quarter of the tiles
    launch = min(tiles, appended // 1024 + 1)
    values = max(4864 * launch + (4 << 20), 16384 * min(launch, max(tiles // 4, 8192), 131072))
    selected = 8 * appended + 48 * N
    return int(psi + core + tables + plan + staging + pool + lists + spilled + values + selected
               + (64 << 20))


def _least(norb, ndets, C, N, batch_pairs):
    """What a request must fit the budget with: the staging of a batch that fills its cap,
    the candidate pool, the psi tables, the item lists and the integral tables."""
    return int(28 * batch_pairs + 32 * (N + min(batch_pairs, 1 << 29)) + 48 * ndets
               + 40 * norb ** 4 + 64 * C * (1 + norb * norb) + (64 << 20))


def _shape(torch, dets):
    """What footprint() can know of a determinant list beside its length."""
    a, b = (bin(int(x)).count("1") for x in dets[0])
    if a + b == 0:
        return {}
    count = torch.unique(dets[:, 0], return_counts=True)[1]
    return dict(na=a, nb=b, alphas=int(count.numel()), group=int(count.max()))


class Server:
    """Search requests against resident systems, continuously batched.

    ``slots``: searches in flight at most; ``budget``: device bytes the running
    searches may hold together (default: half the free memory at start);
    ``search_fn``: the search call (the library's by default; tests may pass a
    stand-in with the same signature).
    """

    def __init__(self, slots: int = 8, budget: int | None = None, search_fn=None):
        import torch
        self._torch = torch
        self._fn = search_fn or _search
        if budget is None:
            free, _ = torch.cuda.mem_get_info()
            budget = free // 2
        self.budget = int(budget)
        self.slots = int(slots)
        self._systems = {}
        self._pending = collections.deque()
        self._cv = threading.Condition()
        self._in_use = 0
        self._running = 0
        self._closed = False
        self.peak_bytes = 0
        self.peak_running = 0
        self.cancelled = 0  # requests withdrawn before admission
        self._workers = [threading.Thread(target=self._work, daemon=True) for _ in range(slots)]
        for t in self._workers:
            t.start()

    # -------------------------------------------------------------- systems ---
    def register(self, name, dets, coeffs, E0, h1, eri, ecore):
        """Keep a system resident (inputs are copied to the device once)."""
        torch = self._torch
        dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")

        def dv(x, dt):
            return x.to(dev) if hasattr(x, "to") else torch.tensor(np.asarray(x), dtype=dt, device=dev)

        d = dets if hasattr(dets, "to") else torch.tensor(np.asarray(dets).astype(np.int64))
        h = dv(h1, torch.float64)
        self._systems[name] = dict(dets=d.to(dev), coeffs=dv(coeffs, torch.float64), E0=float(E0),
                                   h1=h, eri=dv(eri, torch.float64), ecore=float(ecore),
                                   norb=int(round(h.numel() ** 0.5)), ndets=int(d.shape[0]),
                                   shape=_shape(torch, d))

    # ------------------------------------------------------------- requests ---
    def submit(self, name, C: int, N: int, precision: int = FP64, batch_pairs: int = 1 << 26):
        """Queue a search of system ``name``; returns a Future of
        (dets, scores, stats, latency_s) with latency from submission.  A
        request still in the queue is withdrawn by the future's cancel()
        (which then returns True); one already admitted runs to its end."""
        sy = self._systems[name]
        fp = footprint(sy["norb"], sy["ndets"], C, N, batch_pairs, **sy["shape"])
        need = _least(sy["norb"], sy["ndets"], C, N, batch_pairs)
        if need > self.budget:
            raise ValueError(f"request needs {need} bytes, more than the budget {self.budget}")
        fp = min(fp, self.budget)  # an upper estimate beyond the budget: it runs alone
        fut = Future()
        fut.add_done_callback(self._on_done)
        with self._cv:
            if self._closed:
                raise RuntimeError("server closed")
            self._pending.append((name, C, N, precision, batch_pairs, fp, fut, time.perf_counter()))
            self._cv.notify_all()
        return fut

    def _on_done(self, fut):
        # a withdrawn request may have been the one holding up the queue
        if fut.cancelled():
            with self._cv:
                self._cv.notify_all()

    def close(self):
        with self._cv:
            self._closed = True
            self._cv.notify_all()
        for t in self._workers:
            t.join()

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.close()

    # -------------------------------------------------------------- workers ---
    def _next(self):
        """The oldest pending request, once it fits the budget (arrival order:
        a large request is not overtaken indefinitely)."""
        with self._cv:
            while True:
                # withdrawn requests leave the queue without taking a slot
                while self._pending and self._pending[0][6].cancelled():
                    self._pending.popleft()
                    self.cancelled += 1
                if self._pending:
                    fp = self._pending[0][5]
                    if self._in_use + fp <= self.budget:
                        req = self._pending.popleft()
                        if not req[6].set_running_or_notify_cancel():  # withdrawn just now
                            self.cancelled += 1
                            continue
                        self._in_use += fp
                        self._running += 1
                        self.peak_bytes = max(self.peak_bytes, self._in_use)
                        self.peak_running = max(self.peak_running, self._running)
                        return req
                elif self._closed:
                    return None
                self._cv.wait()

    def _work(self):
        torch = self._torch
        stream = torch.cuda.Stream() if torch.cuda.is_available() else None
        while True:
            req = self._next()
            if req is None:
                return
            name, C, N, prec, bp, fp, fut, t0 = req
            sy = self._systems[name]
            try:
                if stream is not None:
                    with torch.cuda.stream(stream):
                        od, osc, st = self._fn(sy["dets"], sy["coeffs"], sy["E0"], sy["h1"],
                                               sy["eri"], sy["ecore"], C, N, precision=prec,
                                               max_batch_pairs=bp, stream=stream)
                        stream.synchronize()
                else:
                    od, osc, st = self._fn(sy["dets"], sy["coeffs"], sy["E0"], sy["h1"], sy["eri"],
                                           sy["ecore"], C, N, precision=prec, max_batch_pairs=bp,
                                           stream=None)
                fut.set_result((od, osc, st, time.perf_counter() - t0))
            except Exception as e:  # reported through the future
                fut.set_exception(e)
            finally:
                with self._cv:
                    self._in_use -= fp
                    self._running -= 1
                    self._cv.notify_all()
