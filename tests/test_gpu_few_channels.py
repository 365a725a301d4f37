"""Layers of few channels on the CUDA cores: rows of one to five vectors among the zeros of the dropped rows, and forwards with short
reductions at the edges of their tiles, against the oracle."""
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


@pytest.mark.parametrize("dtype,M,C_in,C_out,flags", [
    ("f32", 1, 4, 4, 0), ("f32", 65, 12, 68, 0), ("f32", 129, 16, 4, 64), ("f32", 200, 20, 196, 64), ("f32", 64, 48, 64, 0), ("f32", 63, 44, 60, 64),
    ("f32", 20000, 40, 36, 0), ("f32", 20001, 36, 132, 64), ("f32", 80000, 64, 8, 0), ("f32", 40000, 28, 128, 0), ("f32", 7000, 64, 192, 0),
    ("bf16", 3, 8, 8, 0), ("bf16", 784, 16, 64, 64), ("bf16", 513, 24, 24, 0), ("bf16", 200, 32, 256, 64), ("bf16", 20000, 48, 16, 0),
    ("bf16", 16385, 40, 8, 64), ("bf16", 12545, 16, 200, 0), ("bf16", 196, 8, 4096, 0), ("bf16", 300, 64, 40, 8),
])
def test_forward_with_short_reductions(dtype, M, C_in, C_out, flags):
    X, W, _ = synth.layer_inputs(dtype, M, C_in, C_out, 82)
    bias = np.linspace(-1, 1, C_out, dtype=np.float32)
    want = oracle.linear_forward(synth.to_f64(X, dtype), synth.to_f64(W, dtype), bias)
    W_d = dev(np.ascontiguousarray(W.T) if flags & sbp.SBP_FLAG_W_OUT_IN else W, dtype)
    X_d = dev(X, dtype)
    Y = torch.full((M, C_out), float("nan"), dtype=X_d.dtype, device="cuda")
    sbp.sbp_linear_forward(dt_code(dtype), X_d, W_d, torch.from_numpy(bias).cuda(), M, C_in, C_out, Y, flags=flags)
    torch.cuda.synchronize()
    got = synth.to_f64(host(Y), dtype)
    # one rounding of the output, and sums of at most 64 fp32 products
    bound = (2.0 ** -8 if dtype == "bf16" else 0.0) * np.abs(want) + 1e-5 * np.abs(want).max()
    assert (np.abs(got - want) <= bound).all()
