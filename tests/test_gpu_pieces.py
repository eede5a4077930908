"""Pieces and claims of the emission's runs (-m gpu): o = 0 runs shorter than, equal to
and longer than a piece, with a ragged last chunk, in batches of every size class."""
import numpy as np
import pytest

import workloads as W
from tests._parity import compare_candidates, to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb,nd", [(9, 2, 4, 40), (12, 1, 3, 30), (14, 2, 7, 60), (16, 1, 8, 300)])
def test_runs_in_pieces(oracle_mod, n, na, nb, nd):
    """Beta singles and doubles of one determinant: 80, 135, 490 and 848 pairs; few alpha
    strings, so that nearly every pair belongs to such a run and most cells are hot."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    h1, eri, _ = W.random_molecular(n, 60 + n)
    rng = np.random.default_rng(n)
    alphas = [(1 << na) - 1, ((1 << na) - 1) << 1]
    betas = sorted({int(sum(1 << int(q) for q in rng.choice(n, nb, replace=False)))
                    for _ in range(3 * nd)})[:nd // 2]
    A = np.repeat(np.array(alphas, np.uint64), len(betas))
    B = np.tile(np.array(betas, np.uint64), 2)
    c = W.rank_decay_coeffs(len(A), n)
    ints = oracle_mod.Ints(h1, eri, 0.5)
    E0 = min(oracle_mod.diag(ints, (int(a), int(b))) for a, b in zip(A, B)) - 20.0
    dev = lambda x: torch.tensor(x, device="cuda")
    d, s, st = asci.search(dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri),
                           0.5, len(A), 10 ** 6)
    ga, gb = to_u64_pairs(d)
    ref = oracle_mod.search(ints, A, B, c, E0, len(A))
    assert st.generated == ref.generated
    compare_candidates(ga, gb, s.cpu().numpy(), ref, E0, st.diag_grid_bits, label=f"pieces {n}")
