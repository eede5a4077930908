"""The selection's digit rounds and the one-CTA sort (-m gpu) at the sizes and values
where they change: ties that only the key words settle, zeros, subnormals and
infinities among the scores; list lengths around a warp, a CTA and a tile."""
import numpy as np
import pytest

from tests._parity import to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _dev(torch, a, b):
    return torch.tensor(np.stack([a, b], 1).astype(np.int64), device="cuda")


@pytest.mark.parametrize("kind", ["equal", "zeros", "extremes", "two values", "close"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 257, 4097, 30_011])
def test_select_topn_edges(torch_cuda, oracle_mod, kind, n):
    import paper_2303_05688_gb300 as asci
    rng = np.random.default_rng(n)
    key = rng.permutation(np.unique(rng.integers(0, 1 << 62, 2 * n).astype(np.uint64)))[:n]
    a, b = key & np.uint64(0xFFFFFFFF), key >> np.uint64(32)
    s = {"equal": np.full(n, -0.75),
         "zeros": np.where(rng.random(n) < 0.5, 0.0, -0.0),
         "extremes": rng.choice([0.0, 5e-324, -2e-310, 1e308, -np.inf, np.inf, 1.0], n),
         "two values": rng.choice([1.0, -(1.0 + 2.0 ** -52)], n),
         "close": 1.0 + rng.integers(0, 1 << 20, n) * 2.0 ** -52}[kind]
    for N in sorted({1, 2, n // 3 + 1, n - 1, n, n + 3} - {0}):
        k, sc = asci.select_topn(_dev(torch_cuda, a, b), torch_cuda.tensor(s, device="cuda"), N)
        ga, gb = to_u64_pairs(k)
        i = oracle_mod.topn(a, b, s, N)
        assert set(zip(ga.tolist(), gb.tolist())) == set(zip(a[i].tolist(), b[i].tolist()))
        of = dict(zip(zip(a.tolist(), b.tolist()), s.tolist()))
        assert [of[t] for t in zip(ga.tolist(), gb.tolist())] == sc.cpu().numpy().tolist()


@pytest.mark.parametrize("n", [2, 31, 32, 33, 255, 256, 257, 511, 513, 3840, 4095, 4096, 4097])
@pytest.mark.parametrize("bits", [1, 9, 31])
def test_small_sort_is_stable(torch_cuda, n, bits):
    """Equal keys keep their input order: the sums are those of adding in that order, bit
    for bit."""
    import paper_2303_05688_gb300 as asci
    rng = np.random.default_rng(100 * n + bits)
    a = rng.integers(0, 1 << bits, n).astype(np.uint64)
    b = rng.integers(0, 2, n).astype(np.uint64) << np.uint64(31)
    v = rng.normal(size=n) * 10.0 ** rng.integers(-8, 8, n)
    k, s = asci.sort_accumulate(_dev(torch_cuda, a, b), torch_cuda.tensor(v, device="cuda"))
    ga, gb = to_u64_pairs(k)
    key = (b << np.uint64(32)) | a
    uk, inv = np.unique(key, return_inverse=True)
    ref = np.zeros(len(uk))
    np.add.at(ref, inv, v)  # in input order
    assert np.array_equal((gb << np.uint64(32)) | ga, uk)
    assert np.array_equal(s.cpu().numpy(), ref)
