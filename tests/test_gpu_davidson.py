"""Davidson's subspace eigensolve and fused passes (-m gpu) on dense matrices handed
over as CSR: every subspace size class, sizes around a block, restarts, and lowest
eigenvalues too close for FP32 to tell apart.  For a symmetric A and a unit v with
|A v - E v| <= tol, some eigenvalue lies within tol of E."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(n, spread, seed):
    rng = np.random.default_rng(seed)
    w = np.sort(rng.uniform(0.0, 8.0, n)) - 3.0
    w[: min(3, n)] = -20.0 + spread * np.arange(min(3, n))
    q, _ = np.linalg.qr(np.eye(n) + 0.02 * rng.normal(size=(n, n)))
    a = (q * w) @ q.T
    return (a + a.T) / 2, w


@pytest.mark.parametrize("n,sub,spread", [
    (1, 2, 1.0), (2, 2, 1.0), (3, 2, 1.0), (5, 32, 1.0), (16, 16, 0.5), (17, 17, 0.5), (33, 32, 0.5),
    (127, 3, 0.5), (128, 8, 0.5), (129, 9, 0.5), (300, 15, 0.25), (300, 16, 0.25), (700, 31, 0.25),
    (300, 16, 0.0), (300, 16, 1e-13), (300, 16, 1e-10), (300, 24, 1e-7), (300, 8, 1e-5),
])
def test_davidson_subspace(n, sub, spread):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    a, w = _matrix(n, spread, 7 * n + sub)
    rp = torch.arange(0, n * n + 1, n, dtype=torch.int64, device="cuda")
    col = torch.arange(n, dtype=torch.int32, device="cuda").repeat(n)
    val = torch.tensor(a.reshape(-1), device="cuda")
    tol = 1e-9
    guess = torch.tensor(np.random.default_rng(n).normal(size=n), device="cuda")
    for g in (None, guess):
        e, v, it, res = asci.davidson((rp, col, val), g, max_subspace=sub, max_iter=3000, tol=tol)
        v = v.cpu().numpy()
        norm_a = np.abs(a).sum(1).max()
        round_off = 64 * np.finfo(float).eps * norm_a  # of the residual's own formation
        assert abs(np.linalg.norm(v) - 1) < 1e-12
        assert np.linalg.norm(a @ v - e * v) <= tol + round_off
        assert abs(e - w[0]) <= tol + round_off + 2 * spread * (spread < 1e-6)
        assert v[np.argmax(np.abs(v))] > 0
        # the same call gives the same bits
        e2, v2, it2, _ = asci.davidson((rp, col, val), g, max_subspace=sub, max_iter=3000, tol=tol)
        assert e2 == e and it2 == it and np.array_equal(v2.cpu().numpy(), v)
