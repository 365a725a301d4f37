"""Random masks of large maps against the oracle: bins with more words than are ranked directly, slices of a cluster that end inside a
warp's stretch, and masks that keep every position."""
import numpy as np
import pytest

import oracle
import paper_2210_00129_b200 as sbp
from gpu_harness import host, run_sample_keep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,r,flags", [
    (3, 98304, 1, 0.5, 0), (2, 100003, 1, 0.1, 0), (5, 200000, 1, 0.9, 0), (75, 50001, 1, 0.5, 0), (1, 700001, 1, 0.3, 0),
    (2, 333, 201, 0.999, 0), (1, 8193, 1, 0.0001, 0), (4, 513, 1, 0.5, sbp.SBP_FLAG_SHARE_MASK),
    (2, 200, 334, 1.0, 0), (7, 7, 7, 1.0, sbp.SBP_FLAG_SHARE_MASK), (700, 3, 5, 1.0, 0), (1, 1, 1, 1.0, 0), (3, 1, 2, 0.8, 0),   # K = N
])
def test_large_maps_and_full_masks(B, H, W, r, flags):
    rows, offs, cap = run_sample_keep(0, B, H, W, r, seed=11, step=3, offset=2, flags=flags)
    keep, want_offs = oracle.sample_keep(0, B, H, W, r, 11, 3, 2, flags)
    assert np.array_equal(host(offs), want_offs)
    assert np.array_equal(host(rows)[:len(keep)], keep)
