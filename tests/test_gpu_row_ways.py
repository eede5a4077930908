"""The Hamiltonian build's two ways to a row's determinants a beta double away (-m gpu): by
the determinants of its alpha string, or by searching that string in the groups a double
away, whichever is less work.  Each list is built and compared with the oracle, and the
way it took is read from the trace."""
import itertools
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _strings(n, k):
    return np.array([sum(1 << i for i in c) for c in itertools.combinations(range(n), k)], np.uint64)


def determinants(kind):
    """(orbitals, alphas, betas, way)"""
    if kind == "walk":
        A, B = W.random_walk_dets(14, 5, 6, 1500, 9)
        return 14, A, B, "mates"
    n, a, b, way = {
        # one alpha string: as many mates as determinants
        "one alpha": (12, _strings(12, 5)[:1], _strings(12, 4), "searches"),
        "two alphas": (12, _strings(12, 5)[[0, 400]], _strings(12, 5), "searches"),
        # many of few
        "few betas": (12, _strings(12, 5), _strings(12, 4)[[0, 3, 77]], "mates"),
        # the betas of a few orbitals among many: more doubles than as many of all
        # strings would have, so the count of pairs turns the choice
        "a corner": (20, _strings(20, 3)[[0, 5, 500]], _strings(8, 4), "mates"),
        "no doubles": (12, _strings(12, 5)[:40], _strings(12, 1), "mates"),
    }[kind]
    return n, np.repeat(a, len(b)), np.tile(b, len(a)), way


_RUN = """
import sys, numpy as np, torch
import paper_2303_05688_gb300 as asci, workloads as W, oracle
from tests.test_gpu_row_ways import determinants
n, A, B, _ = determinants(sys.argv[1])
h1, eri, ec = W.random_molecular(n, 6)
ref = oracle.dense_h(oracle.Ints(h1, eri, ec), A, B)
for order in (np.lexsort((A, B)), np.random.default_rng(1).permutation(len(A))):
    dets = torch.tensor(np.stack([A[order], B[order]], 1).astype(np.int64), device="cuda")
    rp, col, val = (t.cpu().numpy() for t in asci.hamiltonian(dets, h1, eri, ec))
    want, got = ref[np.ix_(order, order)], np.zeros_like(ref)
    for r in range(len(A)):
        c = col[rp[r]:rp[r + 1]]
        assert np.all(np.diff(c) > 0)
        got[r, c] = val[rp[r]:rp[r + 1]]
    assert np.allclose(got, want, rtol=1e-12, atol=1e-12)
    assert np.all(got[np.abs(want) > 1e-12] != 0.0)
print("AGREE")
"""


@pytest.mark.parametrize("kind", ["walk", "one alpha", "two alphas", "few betas", "a corner",
                                  "no doubles"])
def test_ways(oracle_mod, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _RUN, kind], cwd=root, capture_output=True, text=True,
                       env=dict(os.environ, ASCI_TRACE="1", PYTHONPATH=root), timeout=300)
    assert r.returncode == 0 and "AGREE" in r.stdout, r.stderr[-2000:]
    ways = set(re.findall(r"hamiltonian rows: .* by (\w+)", r.stderr))
    assert ways == {determinants(kind)[3]}
