"""The tile kernel's value buffers (-m gpu): a launch whose buffers are too small
is run again with room for every record, with the same results."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_RUN = """
import numpy as np, torch, sys
import workloads as W, paper_2303_05688_gb300 as asci
w = W.WORKLOADS["random_16e16o"]
h1, eri, ec = w.integrals()
A, B, c = w.psi()
C, N, eps, cap = int(sys.argv[1]), int(sys.argv[2]), float(sys.argv[3]), int(sys.argv[4])
dev = lambda x: torch.tensor(x, device="cuda")
args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(c), W.stored_e0(w.name), dev(h1), dev(eri),
        ec, C, N)
small = asci.search(*args, eps=eps, max_batch_pairs=cap, sort_output=True)
print("SMALL DONE", file=sys.stderr, flush=True)
whole = asci.search(*args, eps=eps, sort_output=True)
assert small[2].batches > whole[2].batches
for k in (0, 1):
    assert torch.equal(small[k], whole[k])
for name in ("surviving", "unique", "excluded", "selected"):
    assert getattr(small[2], name) == getattr(whole[2], name), name
print("AGREE", len(small[1]))
"""


@pytest.mark.parametrize("C,N,eps,cap,full", [
    (4000, 2_500_000, 0.0, 1 << 22, True),    # a low threshold: half of all targets reach it
    (4000, 2_500_000, 1e-8, 1 << 22, True),   # with records dropped by the screen
    (4000, 1_000, 0.0, 1 << 22, False),       # an ordinary threshold fits the buffers
])
def test_value_buffers(C, N, eps, cap, full):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _RUN, str(C), str(N), str(eps), str(cap)], cwd=root,
                       env=dict(os.environ, ASCI_TRACE="1", PYTHONPATH=root), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "AGREE" in r.stdout, r.stderr[-2000:]
    first = r.stderr.split("SMALL DONE")[0]
    assert ("values found no room" in first) == full
