"""Davidson's lowest root among two that FP32 cannot tell apart (-m gpu)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [1e-4, 1e-6, 1e-7, 3e-8])
def test_the_lower_of_two_near_values(split):
    """Tridiagonal matrices: a random block, and one element below its lowest eigenvalue by
    `split`, linked to the block's end by 1e-13.  From the first unit vector every
    correction is the next unit vector, so the last product's subspace is the whole space
    and the result the lowest eigenvalue of the matrix."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    dev = lambda x, t: torch.tensor(x, dtype=t, device="cuda")
    wrong = []
    for seed in range(200):
        rng = np.random.default_rng(seed)
        n = int(rng.integers(4, 10))
        t = np.diag(rng.uniform(-1.0, 8.0, n))
        off = rng.uniform(0.5, 2.0, n - 1)
        off[-1] = 1e-13
        t += np.diag(off, 1) + np.diag(off, -1)
        t[-1, -1] = np.linalg.eigvalsh(t[:-1, :-1])[0] - split
        at = [(i, j) for i in range(n) for j in (i - 1, i, i + 1) if 0 <= j < n]
        rp = np.searchsorted([i for i, _ in at], np.arange(n + 1))
        e, _, it, _ = asci.davidson(
            (dev(rp, torch.int64), dev([j for _, j in at], torch.int32),
             dev([t[i, j] for i, j in at], torch.float64)),
            dev(np.eye(n)[0], torch.float64), max_subspace=32, tol=1e-30)
        assert it == n
        # eigenvalues of an n x n matrix in FP64, on both sides
        if abs(e - np.linalg.eigvalsh(t)[0]) > 64 * n * np.finfo(float).eps * np.abs(t).sum(1).max():
            wrong.append((seed, e))
    assert not wrong, wrong
