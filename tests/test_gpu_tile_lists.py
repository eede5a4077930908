"""A tile in which every record that one warp claims has further records elsewhere
(-m gpu): 256 targets to be summed in one warp, the most that its counts must hold."""
import itertools

import numpy as np
import pytest

import workloads as W
from tests._parity import compare_candidates, to_u64_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("markers", [0, 32])
def test_a_warp_of_lists(oracle_mod, markers):
    """32 alpha strings, each a double excitation away from the string `to`, with 32 beta
    strings each; the strings 2k and 2k + 1 have the same betas.  The class of `to` is one
    tile of 1024 records in item order, whose records p and p + 32 (of even p // 32) share
    a target: of each such pair of warps, the one that is first claims up to 256 targets of
    two records.  Determinants of psi that fall in the tile hold back its first warp."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    n, to = 12, 0b111111
    h1, eri, _ = W.random_molecular(n, 21)
    alphas = sorted(to ^ (1 << i) ^ (1 << j) ^ (1 << a) ^ (1 << b)
                    for i, j in itertools.combinations(range(6), 2)
                    for a, b in itertools.combinations(range(6, 12), 2))[::7][:32]
    betas = [sum(1 << i for i in c) for c in itertools.combinations(range(n), 6)]
    pick = np.random.default_rng(3).permutation(len(betas))
    core = [(a, betas[pick[32 * (k // 2) + j]]) for k, a in enumerate(alphas) for j in range(32)]
    psi = core + [(to, betas[pick[512 + j]]) for j in range(markers)]
    A, B = (np.array(x, np.uint64) for x in zip(*psi))
    c = np.where(np.arange(len(psi)) % 3 == 0, -1.0, 1.0) / np.arange(30, 30 + len(psi))
    c /= np.linalg.norm(c)
    ints = oracle_mod.Ints(h1, eri, 0.5)
    E0 = min(oracle_mod.diag(ints, (int(a), int(b))) for a, b in psi) - 20.0
    dev = lambda x: torch.tensor(x, device="cuda")
    args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, dev(h1), dev(eri), 0.5, len(core),
            10 ** 6)
    ref = oracle_mod.search(ints, A, B, c, E0, len(core))
    assert int((ref.a == to).sum()) >= 512  # the tile's targets
    first = None
    for _ in range(5):
        d, s, st = asci.search(*args, sort_output=True)
        if first is None:
            first = (d, s)
            ga, gb = to_u64_pairs(d)
            assert st.unique == ref.unique
            compare_candidates(ga, gb, s.cpu().numpy(), ref, E0, st.diag_grid_bits,
                               label=f"a warp of lists {markers}")
        assert torch.equal(d, first[0]) and torch.equal(s, first[1])
