"""`sbp_sample_keep` where its block size, clusters, word cache and stretches (random masks) or its blocks per sample (grid masks)
change, bit for bit against the oracle: one position, one group more or less than the threads, every cluster size, maps beyond the cache, extreme ratios."""
import numpy as np
import pytest

import oracle
from gpu_harness import run_sample_keep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,r", [
    (3, 1, 1, 0.5), (2, 1, 3, 0.34), (2, 1, 5, 1.0), (300, 1, 196, 0.25), (2, 1, 511, 0.5), (2, 1, 512, 0.999), (2, 1, 513, 0.001),
    (3, 1, 2047, 0.5), (3, 1, 2049, 0.5), (2, 1, 8192, 0.5), (2, 1, 8193, 0.5), (5, 1, 16385, 0.1), (3, 1, 32769, 0.9), (1, 1, 32773, 1e-5),
    (2, 200, 334, 0.5), (4, 1, 32771, 0.5), (3, 1, 70001, 0.999), (80, 1, 8197, 0.5), (76, 1, 41003, 0.3), (1, 3, 100001, 0.5), (1, 1000, 1000, 0.25),
])
def test_random_masks_at_every_dispatch(B, H, W, r):
    for share in (0, 1):
        rows, offs, cap = run_sample_keep(0, B, H, W, r, seed=9 + share, step=3, offset=2, flags=share)
        keep, want_offs = oracle.sample_keep(0, B, H, W, r, 9 + share, 3, 2, bool(share))
        assert np.array_equal(offs.cpu().numpy(), want_offs)
        assert np.array_equal(rows.cpu().numpy()[:len(keep)], keep)


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (3, 1, 7), (3, 7, 1), (2, 45, 46), (70, 7, 7), (600, 3, 5), (2, 200, 334), (3, 333, 201), (1, 1024, 1025)])
def test_grid_masks_at_every_split(B, H, W):
    for r in (0.25, 0.5, 0.75, 1.0):
        for share in (0, 1):
            rows, offs, cap = run_sample_keep(1, B, H, W, r, seed=9 + share, step=3, offset=2, flags=share)
            keep, want_offs = oracle.sample_keep(1, B, H, W, r, 9 + share, 3, 2, bool(share))
            assert np.array_equal(offs.cpu().numpy(), want_offs)
            assert np.array_equal(rows.cpu().numpy()[:len(keep)], keep)


@pytest.mark.parametrize("B,T,P", [(1, 1, 1), (1, 8, 196), (3, 7, 1), (2, 33, 1000), (600, 5, 9), (1, 2048, 3), (2, 64, 3136)])
@pytest.mark.parametrize("mode", [2, 3])
def test_frame_masks_at_every_split(mode, B, T, P):
    for r in (0.25, 0.5, 0.75):
        for share in (0, 1):
            rows, offs, cap = run_sample_keep(mode, B, T, P, r, seed=9 + share, step=3, offset=2, flags=share)
            keep, want_offs = oracle.sample_keep(mode, B, T, P, r, 9 + share, 3, 2, bool(share))
            assert np.array_equal(offs.cpu().numpy(), want_offs)
            assert np.array_equal(rows.cpu().numpy()[:len(keep)], keep)
