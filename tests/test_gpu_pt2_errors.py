"""ASCI-PT2 with a vanishing denominator among the targets of any batch (-m gpu): invalid
input, whichever launch finds it."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [0, 1 << 20, 1 << 16])
def test_vanishing_denominator_before_the_last_batch(cap):
    """On the ring, the same-occupancy doubles of the aufbau determinant have its H_ii."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2303_05688_gb300 as asci
    h1, eri, ec = W.hubbard_ring(12, 1.0, 4.0)
    A, B = W.random_walk_dets(12, 6, 6, 4000, 5)
    c = W.rank_decay_coeffs(4000, 5)
    E0 = float(np.trace(h1[:6, :6]) * 2 + 6 * 4.0)
    dev = lambda x: torch.tensor(x, device="cuda")
    args = (dev(np.stack([A, B], 1).astype(np.int64)), dev(c), E0, h1, eri, ec, 4000)
    with pytest.raises(asci.AsciError, match="PT2 term") as err:
        asci.pt2(*args, max_batch_pairs=cap)
    assert "ASCI_EINVAL" in str(err.value)
    e, st = asci.pt2(*args[:2], E0 - 40.0, *args[3:], max_batch_pairs=cap)  # later calls run
    assert np.isfinite(e) and (cap == 0 or st.batches > 1)
