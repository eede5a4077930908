"""The radix sort over tiles (-m gpu): stability and order at lengths around one, two and
many tiles, where the tiles' wait for one another is shortest and longest, and with keys
that fill every digit, one digit, or one value."""
import numpy as np
import pytest

from tests._parity import to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4097, 8191, 8192, 8193, 100_003, 1_000_001, 5_000_000])
@pytest.mark.parametrize("kind", ["wide", "one digit", "two values", "sorted", "reversed"])
def test_sort_over_tiles(n, kind):
    """Sums of equal keys are those of adding in input order, bit for bit, so they show a
    key or a value out of place."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    rng = np.random.default_rng(n)
    key = {"wide": lambda: rng.integers(0, 1 << 63, n, dtype=np.uint64),
           "one digit": lambda: rng.integers(0, 256, n, dtype=np.uint64) << np.uint64(40),
           "two values": lambda: np.where(rng.random(n) < 1e-4, np.uint64(1), np.uint64(1) << np.uint64(50)),
           "sorted": lambda: np.arange(n, dtype=np.uint64) // np.uint64(3),
           "reversed": lambda: np.arange(n, dtype=np.uint64)[::-1] * np.uint64(1 << 20)}[kind]()
    key = np.ascontiguousarray(key, dtype=np.uint64)
    v = rng.normal(size=n) * 10.0 ** rng.integers(-8, 8, n)
    dets = torch.tensor(np.stack([key & np.uint64(0xFFFFFFFF), key >> np.uint64(32)], 1).astype(np.int64),
                        device="cuda")
    k, s = asci.sort_accumulate(dets, torch.tensor(v, device="cuda"))
    ga, gb = to_u64_pairs(k)
    uk, inv = np.unique(key, return_inverse=True)
    ref = np.zeros(len(uk))
    np.add.at(ref, inv, v)  # in input order
    assert np.array_equal((gb << np.uint64(32)) | ga, uk)
    assert np.array_equal(s.cpu().numpy(), ref)
