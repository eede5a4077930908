"""The eps screen's 32-bit denominators (-m gpu): every pair is decided as by the FP64
test on the exact denominator, also when the threshold lies between a pair's ratio and
the bounds of its 32-bit denominator, and when the denominator is smaller than those
bounds' distance."""
import numpy as np
import pytest

import workloads as W
from tests._parity import grid_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [(6, 3, 3), (9, 4, 3), (17, 2, 3)])
@pytest.mark.parametrize("where", ["below", "inside"])
def test_eps_next_to_pairs(oracle_mod, n, na, nb, where):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    h1, eri, _ = W.random_molecular(n, 40 + n)
    A, B = W.random_walk_dets(n, na, nb, 20, n)
    c = W.rank_decay_coeffs(20, n)
    ints = oracle_mod.Ints(h1, eri, 0.5)
    ta, tb, v = oracle_mod.pairs(ints, A, B, c)
    t = list(zip(ta.tolist(), tb.tolist()))
    hd = {d: oracle_mod.diag(ints, d) for d in set(t)}
    hii = np.array([hd[d] for d in t])
    # "inside": 1e-7 off one target's diagonal, closer than the 32-bit sums resolve
    E0 = hii.min() - 1.0 if where == "below" else float(np.median(hii)) + 1e-7
    q = np.abs(v / (E0 - hii))
    order = np.argsort(q)
    dev = lambda x: torch.tensor(x, device="cuda")
    args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri), 0.5)
    checked = 0
    for f in (0.1, 0.5, 0.9, 0.999):
        for side in (-1.0, 1.0):
            # far below the 32-bit sums' resolution, far above FP64 rounding
            eps = float(q[order[int(f * len(q))]]) * (1.0 + side * 3e-10)
            st = asci.search(*args, 20, 10 ** 6, eps=eps)[2]
            # the two sides' errors of E0 - H_ii (grid of the exact sums, FP64 rounding
            # of at most 100 terms below 100) leave the decision to neither
            err = (grid_err(st.diag_grid_bits, na, nb) + 1e-12) / np.abs(E0 - hii) + 1e-14
            if (np.abs(q / eps - 1.0) <= err).any():
                continue
            checked += 1
            assert st.surviving == int((q > eps).sum()), (f, side)
            assert st.surviving == oracle_mod.search(ints, A, B, c, E0, 20, eps=eps).surviving
    assert checked >= 6
