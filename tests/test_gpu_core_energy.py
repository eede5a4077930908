"""Large core energies (-m gpu): the emission's 32-bit denominators resolve E0 - H_ii, in
which the core energy cancels, so a search's work does not depend on it."""
import time

import numpy as np
import pytest

import workloads as W
from tests._parity import compare_candidates, to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _search(torch, h1, eri, ecore, A, B, c, E0, *args, **kw):
    import paper_2303_05688_gb300 as asci
    dev = lambda x: torch.tensor(x, device="cuda")
    return asci.search(dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri), ecore,
                       *args, **kw)


@pytest.mark.parametrize("ecore,below", [(0.0, 1.0), (-3000.0, 1.0), (1e6, 1.0), (1e6, 1e5), (0.0, 1e6)])
@pytest.mark.parametrize("eps", [0.0, 1e-8])
def test_candidates_with_a_core_energy(torch_cuda, oracle_mod, ecore, below, eps):
    """E0 `below` the lowest diagonal: near it, and further than the sum of all terms."""
    n = 10
    h1, eri, _ = W.random_molecular(n, 12)
    A, B = W.random_walk_dets(n, 4, 5, 80, 6)
    c = W.rank_decay_coeffs(80, 6)
    ints = oracle_mod.Ints(h1, eri, ecore)
    E0 = min(oracle_mod.diag(ints, (int(a), int(b))) for a, b in zip(A, B)) - below
    ref = oracle_mod.search(ints, A, B, c, E0, 80, eps=eps)
    d, s, st = _search(torch_cuda, h1, eri, ecore, A, B, c, E0, 80, 10 ** 6, eps=eps)
    assert st.surviving == ref.surviving
    ga, gb = to_u64_pairs(d)
    compare_candidates(ga, gb, s.cpu().numpy(), ref, E0, st.diag_grid_bits,
                       label=f"ecore {ecore:g} below {below:g} eps {eps:g}")


@pytest.mark.parametrize("eps", [0.0, 1e-6])
def test_a_core_energy_costs_no_time(torch_cuda, eps):
    h1, eri, _ = W.random_molecular(30, 7)
    A, B = W.random_walk_dets(30, 12, 12, 20_000, 7)
    c = W.rank_decay_coeffs(20_000, 7)

    def best(ecore):
        t = []
        for _ in range(6):
            torch_cuda.cuda.synchronize()
            t0 = time.perf_counter()
            _search(torch_cuda, h1, eri, ecore, A, B, c, 60.0 + ecore, 3000, 50_000, eps=eps)
            torch_cuda.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(1e9) < 1.5 * best(0.0)
