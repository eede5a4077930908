"""The Hamiltonian build's two merged lists (-m gpu): determinant lists in which a row has
no, one, fewer and more than 32 mates of its own alpha string, in windows with and without
a double among them, against few, many and no neighbouring beta groups."""
import itertools

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _strings(n, k):
    return np.array([sum(1 << i for i in c) for c in itertools.combinations(range(n), k)], np.uint64)


def _product(a, b):
    return np.repeat(a, len(b)), np.tile(b, len(a))


def _lists(kind):
    rng = np.random.default_rng(5)
    if kind == "one alpha":
        return 12, _product(_strings(12, 5)[:1], _strings(12, 4))
    if kind == "one beta":
        return 12, _product(_strings(12, 5), _strings(12, 4)[7:8])
    if kind == "few alphas":
        return 11, _product(rng.choice(_strings(11, 5), 5, replace=False), _strings(11, 5))
    if kind == "few betas":
        return 11, _product(_strings(11, 5), rng.choice(_strings(11, 5), 5, replace=False))
    if kind == "doubles only":  # pairs of orbitals filled together
        p = np.array([sum(3 << (2 * i) for i in c) for c in itertools.combinations(range(7), 3)],
                     np.uint64)
        return 14, _product(p, p)
    A, B = _product(_strings(10, 3), _strings(10, 4))
    keep = np.sort(rng.choice(len(A), {"third": len(A) // 3, "33": 33}[kind], replace=False))
    return 10, (A[keep], B[keep])


@pytest.mark.parametrize("kind", ["one alpha", "one beta", "few alphas", "few betas", "doubles only",
                                  "third", "33"])
@pytest.mark.parametrize("shuffled", [False, True])
def test_merged_rows(oracle_mod, kind, shuffled):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    n, (A, B) = _lists(kind)
    if shuffled:
        order = np.random.default_rng(1).permutation(len(A))
        A, B = A[order], B[order]
    h1, eri, ec = W.random_molecular(n, 6)
    dets = torch.tensor(np.stack([A, B], 1).astype(np.int64), device="cuda")
    rp, col, val = (t.cpu().numpy() for t in asci.hamiltonian(dets, h1, eri, ec))
    ref = oracle_mod.dense_h(oracle_mod.Ints(h1, eri, ec), A, B)
    got = np.zeros_like(ref)
    for r in range(len(A)):
        c = col[rp[r]:rp[r + 1]]
        assert np.all(np.diff(c) > 0)
        got[r, c] = val[rp[r]:rp[r + 1]]
    assert np.allclose(got, ref, rtol=1e-12, atol=1e-12)
    assert np.all(got[np.abs(ref) > 1e-12] != 0.0)
