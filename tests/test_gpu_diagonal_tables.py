"""The exact diagonal by chunk tables (-m gpu): scores and ASCI-PT2 against the
oracle at orbital counts on both sides of every change of the chunk layout (two
chunks up to 16 orbitals, three up to 24, four above; whole and ragged last
chunks)."""
import numpy as np
import pytest

import workloads as W
from tests._parity import compare_candidates, to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [(2, 1, 1), (3, 2, 1), (7, 3, 2), (8, 2, 3), (9, 3, 3), (15, 2, 2),
                                     (16, 2, 2), (17, 2, 2), (23, 2, 1), (24, 2, 2), (25, 2, 2),
                                     (29, 2, 1), (31, 2, 2), (32, 1, 2)])
def test_diagonal_tables(oracle_mod, n, na, nb):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    h1, eri, _ = W.random_molecular(n, 100 + n)
    nd = min(10, W.comb(n, na) * W.comb(n, nb) // 2)
    A, B = W.random_walk_dets(n, na, nb, nd, n)
    c = W.rank_decay_coeffs(nd, n)
    # a determinant that occupies the highest orbitals, so that every chunk is met
    if nd > 2:
        top = (((1 << na) - 1) << (n - na), ((1 << nb) - 1) << (n - nb))
        if top not in set(zip(A.tolist(), B.tolist())):
            A[-1], B[-1] = top
    ints = oracle_mod.Ints(h1, eri, 0.5)
    E0 = min(oracle_mod.diag(ints, (a, b)) for a, b in zip(*W.all_dets(n, na, nb))) - 1.0 \
        if n < 10 else oracle_mod.diag(ints, (int(A[0]), int(B[0]))) - 20.0
    dev = lambda x: torch.tensor(x, device="cuda")
    args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri), 0.5)
    d, s, st = asci.search(*args, nd, 10 ** 6)
    ga, gb = to_u64_pairs(d)
    ref = oracle_mod.search(ints, A, B, c, E0, nd)
    compare_candidates(ga, gb, s.cpu().numpy(), ref, E0, st.diag_grid_bits, label=f"norb {n}")
    e2, e2_ref = asci.pt2(*args)[0], oracle_mod.pt2(ints, A, B, c, E0, nd)
    assert abs(e2 - e2_ref) <= 1e-10 * abs(e2_ref)
