"""The one-pass scan (-m gpu): run positions of sorted keys at lengths around a tile (4096
elements), the 32 tiles of one look back, and many more; row pointers (64-bit sums) of a
matrix whose rows span several tiles."""
import numpy as np
import pytest

import workloads as W
from tests._parity import to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 8192, 131_071, 131_072, 131_073, 135_169, 3_000_001])
@pytest.mark.parametrize("repeat", [1, 2, 5000])
def test_run_positions(torch_cuda, n, repeat):
    import paper_2303_05688_gb300 as asci
    key = np.arange(n, dtype=np.uint64) // np.uint64(repeat)
    dets = torch_cuda.tensor(np.stack([key, np.zeros_like(key)], 1).astype(np.int64), device="cuda")
    k, s = asci.sort_accumulate(dets, torch_cuda.ones(n, dtype=torch_cuda.float64, device="cuda"))
    ga, _ = to_u64_pairs(k)
    uk, cnt = np.unique(key, return_counts=True)
    assert np.array_equal(ga, uk)
    assert np.array_equal(s.cpu().numpy(), cnt.astype(float))


@pytest.mark.parametrize("nd", [4095, 4096, 8193, 20_000])
def test_row_pointers(torch_cuda, nd):
    import paper_2303_05688_gb300 as asci
    h1, eri, ec = W.random_molecular(14, 3)
    A, B = W.random_walk_dets(14, 6, 6, nd, 3)
    dets = torch_cuda.tensor(np.stack([A, B], 1).astype(np.int64), device="cuda")
    rp, col, val = (t.cpu().numpy() for t in asci.hamiltonian(dets, h1, eri, ec))
    assert rp[0] == 0 and rp[-1] == len(col) == len(val)
    lens = np.diff(rp)
    assert lens.min() >= 1
    # symmetric: as many elements in column i as in row i
    assert np.array_equal(np.bincount(col, minlength=len(A)), lens)
    assert np.array_equal(col[[np.flatnonzero(col[rp[i]:rp[i + 1]] == i)[0] + rp[i]
                               for i in range(0, len(A), 97)]], np.arange(0, len(A), 97))
