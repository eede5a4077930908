"""The server's admission with an estimate beyond its budget (CPU, stand-in search)."""
import threading
import time

import numpy as np
import pytest


def test_a_request_beyond_the_budget_runs_alone():
    torch = pytest.importorskip("torch")
    from paper_2303_05688_gb300.serve import Server, footprint
    lock, live, worst = threading.Lock(), [0], [0]

    def fake(dets, coeffs, E0, h1, eri, ecore, C, N, **kw):
        with lock:
            live[0] += 1
            worst[0] = max(worst[0], live[0])
        time.sleep(0.05)
        with lock:
            live[0] -= 1
        return dets[:1], coeffs[:1], {}

    d = np.array([[0b11, 0b101], [0b11, 0b110], [0b101, 0b11]], np.int64)
    shape = dict(na=2, nb=2, alphas=2, group=2)
    budget = footprint(8, 3, 3, 100, 1 << 20, **shape) - 1
    with Server(slots=3, budget=budget, search_fn=fake) as srv:
        srv.register("s", d, np.ones(3), -1.0, np.zeros((8, 8)), np.zeros(8 ** 4), 0.0)
        assert srv._systems["s"]["shape"] == shape
        futs = [srv.submit("s", 3, 100, batch_pairs=1 << 20) for _ in range(3)]
        for f in futs:
            f.result(timeout=30)
    assert worst[0] == 1 and srv.peak_bytes == budget


def test_estimate_grows_with_every_size():
    from paper_2303_05688_gb300.serve import footprint
    shape = dict(na=8, nb=8, alphas=500, group=300)
    sizes = dict(norb=16, ndets=10_000, C=1000, N=1000, batch_pairs=1 << 22)
    base = footprint(**sizes, **shape)
    assert base <= footprint(**sizes)
    for name in sizes:
        assert footprint(**dict(sizes, **{name: 2 * sizes[name]}), **shape) >= base, name
    for name in ("alphas", "group"):
        assert footprint(**sizes, **dict(shape, **{name: 2 * shape[name]})) >= base, name
