"""Layers of few channels on the CUDA cores: rows of one to five vectors among the zeros of the dropped rows, against
the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, dt_code, host, run_backward, run_forward_cache

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C_in", [4, 8, 12, 16, 20, 68])
@pytest.mark.parametrize("M,keep_every", [(700, 20), (33, 33), (5000, 2), (96, 1)])
def test_dropped_rows_of_few_vectors(C_in, M, keep_every):
    C_out = 12
    X, W, dY = synth.layer_inputs("f32", M, C_in, C_out, 81)
    keep = np.arange(0, M, keep_every, dtype=np.int32)
    rows = torch.from_numpy(keep).cuda()
    Xk = run_forward_cache("f32", dev(X, "f32"), rows, len(keep))
    got = run_backward("f32", Xk, dev(dY, "f32"), dev(W, "f32"), rows, len(keep))
    want = oracle.linear_backward(X[keep].astype(np.float64), dY.astype(np.float64), W.astype(np.float64), keep)
    dX = host(got["dX"])
    assert not dX[np.setdiff1d(np.arange(M), keep)].view(np.uint32).any()
    for g, w in ((dX, want["dX"]), (host(got["dW"]), want["dW"]), (host(got["db"]), want["db"])):
        assert np.abs(g - w).max() <= 1e-5 * np.abs(w).max()              # fp32 sums of at most 2500 terms

