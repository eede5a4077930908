"""The server's admission estimate against the memory that searches take from the device
(-m gpu): never less, for ordinary and served sizes, ASCI-PT2, few alpha strings (whose
hot targets overfill their buckets) and the smallest call."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _few_alphas():
    n = 14
    h1, eri, _ = W.random_molecular(n, 5)
    A, B = W.random_walk_dets(n, 7, 7, 40_000, 5)
    keep = np.isin(A, np.unique(A)[:3])
    return h1, eri, A[keep], B[keep]


@pytest.mark.parametrize("n,na,nd,C,N,cap", [
    (30, 12, 4000, 4000, 0, 1 << 26), (30, 12, 200_000, 20_000, 10_000_000, 1 << 26),
    (30, 12, 100_000, 10_000, 100_000, 1 << 22), (16, 8, 50_000, 5000, 2_500_000, 1 << 22),
    (20, 10, 20_000, 20_000, 1_000_000, 1 << 28), (12, 6, 2000, 200, 5000, 1 << 20),
    (8, 4, 100, 100, 1000, 1 << 26), (4, 2, 5, 5, 10, 1 << 26), (14, 7, 0, 0, 1_000_000, 1 << 24),
    (14, 7, 0, 0, 0, 1 << 24),
])
def test_footprint_is_an_upper_estimate(n, na, nd, C, N, cap):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    from paper_2303_05688_gb300.serve import Server, footprint
    if nd:
        h1, eri, _ = W.random_molecular(n, 3)
        A, B = W.random_walk_dets(n, na, na, nd, 3)
    else:
        h1, eri, A, B = _few_alphas()
        nd = C = len(A)
    dev = lambda x: torch.tensor(x, device="cuda")
    d, c, h1, eri = dev(np.stack([A, B], 1).astype(np.int64)), dev(W.rank_decay_coeffs(nd, 3)), dev(h1), dev(eri)
    with Server(slots=1, budget=1 << 50) as srv:
        srv.register("s", d, c, -100.0, h1, eri, 0.0)
        shape = srv._systems["s"]["shape"]
    bound = footprint(n, nd, C, N, cap, **shape)
    assert bound <= footprint(n, nd, C, N, cap)
    asci.load().asci_trim_cache()
    # the outputs' memory is the caller's: taken from torch's cache, filled before
    out = torch.empty(4 * max(N, 1), dtype=torch.int64, device="cuda")
    del out
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    if N:
        asci.search(d, c, -100.0, h1, eri, 0.0, C, N, max_batch_pairs=cap, sort_output=True)
    else:
        asci.pt2(d, c, -100.0, h1, eri, 0.0, C, max_batch_pairs=cap)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    asci.load().asci_trim_cache()
    assert taken <= bound, (taken, bound)
