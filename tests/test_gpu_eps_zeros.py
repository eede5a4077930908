"""The eps screen on pairs of value zero and at thresholds outside the float range (-m gpu):
rings, whose double excitations mostly have no matrix element, and integrals with the
zeros of an orbital symmetry."""
import time

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _symmetric(n, seed):
    """Random integrals that vanish unless the labels of their orbitals (the eight
    representations of D2h) multiply to the first."""
    h1, eri, ec = W.random_molecular(n, seed)
    g = np.random.default_rng(seed).integers(0, 8, n)
    x = g[:, None] ^ g[None, :]
    return np.where(x == 0, h1, 0.0), np.where(x[:, :, None, None] == x[None, None], eri, 0.0), ec


def _system(kind, n):
    return W.hubbard_ring(n, 1.0, 4.0) if kind == "ring" else _symmetric(n, 8)


@pytest.mark.parametrize("kind", ["ring", "symmetric", "random"])
@pytest.mark.parametrize("eps", [1e-3, 1e-10, 1e-40, 1e-300, 5e-324, 1e30])
def test_survivors_with_zeros(torch_cuda, oracle_mod, kind, eps):
    import paper_2303_05688_gb300 as asci
    n = 9
    h1, eri, ec = W.random_molecular(n, 8) if kind == "random" else _system(kind, n)
    A, B = W.random_walk_dets(n, 4, 3, 60, 2)
    c = W.rank_decay_coeffs(60, 2)
    ints = oracle_mod.Ints(h1, eri, ec)
    E0 = min(oracle_mod.diag(ints, (int(a), int(b))) for a, b in zip(A, B)) - 1.0
    ref = oracle_mod.search(ints, A, B, c, E0, 60, eps=eps)
    dev = lambda x: torch_cuda.tensor(x, device="cuda")
    st = asci.search(dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri), ec, 60,
                     10 ** 6, eps=eps)[2]
    assert st.surviving == ref.surviving and st.unique == ref.unique
    if kind != "random" and eps < 1:
        assert st.surviving < st.generated // 3


def test_a_screen_of_zeros_costs_no_more_than_none(torch_cuda):
    """The screen drops these pairs, so a search with it stages less work than one without."""
    import paper_2303_05688_gb300 as asci
    h1, eri, ec = _symmetric(30, 3)
    A, B = W.random_walk_dets(30, 12, 12, 5000, 4)
    dev = lambda x: torch_cuda.tensor(x, device="cuda")
    args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(W.rank_decay_coeffs(5000, 4)), -60.0, dev(h1),
            dev(eri), ec, 2000, 10_000)

    def best(eps):
        t = []
        for _ in range(6):
            torch_cuda.cuda.synchronize()
            t0 = time.perf_counter()
            st = asci.search(*args, eps=eps)[2]
            torch_cuda.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t), st

    with_screen, st = best(1e-10)
    assert st.surviving < st.generated // 4
    assert with_screen < 1.5 * best(0.0)[0]
