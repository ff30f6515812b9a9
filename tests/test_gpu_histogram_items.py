"""Histograms of exit states whose item fields are not all valid: entries of any out-of-range item, sentinels
that wrap a 32-bit difference among them, are not counted wherever they stand, and the others all are."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LN10 = 2.302585092994046


@pytest.mark.parametrize("invalid", [0xFFFFFFFF, 0xFFFFFFF0, 0x80000000, None])
@pytest.mark.parametrize("n_items,nbins", [(30, 512), (16, 512), (5, 512), (3000, 1), (40, 4096), (3, 8190)])
def test_items_out_of_range(n_items, nbins, invalid):
    """The first entry of every 256 (so of every block) is invalid, the next ones valid; None: one above the last."""
    import torch
    n = 40001
    rng = np.random.default_rng(n_items + nbins)
    lnP = rng.normal(1.0, 2.0, n)
    item = np.sort(rng.integers(0, n_items, n)).astype(np.uint32)
    item[n // 2:] = rng.integers(0, n_items, n - n // 2)            # half of them in no order
    item[::256] = n_items if invalid is None else invalid
    out = cz.ExitBuffers(n)
    for t in (out.r, out.th, out.ph, out.s):
        t.fill_(1.0)
    out.steps.fill_(1)
    out.status.fill_(cz.PATH_EXIT)
    out.lnP.copy_(torch.as_tensor(lnP))
    out.item.copy_(torch.as_tensor(item.view(np.int32)))
    # counters on both sides of the histogram show a write beside it
    guard, size = 4096, n_items * (nbins + 3)
    H = torch.full((size + 2 * guard,), -1, dtype=torch.int64, device="cuda")
    J, S = (torch.empty(n_items, dtype=torch.float64, device="cuda") for _ in range(2))
    x_lo, dx = -1.0, 4.0 / nbins
    cz.cosmica_spectrum(out, cz.make_species(W.PROTON), [1.0] * n_items, cz.make_bins(0.1, 1000.0, nbins), J, S,
                        H[guard:guard + size])
    b = np.floor((lnP / LN10 - x_lo) / dx)
    slot = np.where(b < 0, 0, np.where(b >= nbins, nbins + 1, b + 1)).astype(np.int64)
    ok = item < n_items
    want = np.bincount(item[ok].astype(np.int64) * (nbins + 3) + slot[ok], minlength=size)
    got = H.cpu().numpy()
    assert np.array_equal(got[guard:guard + size], want)
    assert np.all(got[:guard] == -1) and np.all(got[guard + size:] == -1)
