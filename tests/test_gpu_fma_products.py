"""The CUDA-core products (fp32, small bf16 layers) at the edges of their tiles and splits, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, dt_code, host, run_backward, run_forward_cache

pytestmark = pytest.mark.gpu


def _check(got, want, dtype, rounded):
    """fp32 sums of n terms: relative error about sqrt(n) 2^-24, below 1e-5 for the sizes here; bf16 outputs: one rounding."""
    g = synth.to_f64(host(got), dtype) if rounded else host(got).astype(np.float64)
    w = np.asarray(want)
    scale = float(np.sqrt(np.mean(w * w)))
    bound = (2.0 ** -8 if rounded and dtype == "bf16" else 1e-5) * np.maximum(np.abs(w), scale) + 1e-5 * scale
    assert (np.abs(g - w) <= bound).all()


@pytest.mark.parametrize("dtype,B,H,W,C_in,C_out,mask,r,accumulate", [
    ("f32", 1, 3, 1, 4, 4, 0, 0.34, False),            # one kept row, one 16-byte vector per row
    ("f32", 3, 11, 7, 60, 132, 0, 0.5, True),          # just below and above a tile; sums into dW and db
    ("f32", 2, 40, 41, 64, 64, 0, 0.9, True),          # dW reduction split over the kept rows, one tile
    ("f32", 2, 12, 49, 68, 260, 2, 0.25, False),       # whole frames: gaps of hundreds of dropped rows
    ("f32", 5, 15, 13, 36, 68, 1, 0.25, False),        # count known on the device only
    ("f32", 4, 14, 25, 1028, 1540, 0, 0.5, False),     # 64 x 128 tiles, ragged in every direction
    ("bf16", 3, 14, 14, 72, 40, 1, 0.75, True),
    ("bf16", 1, 8, 7, 520, 264, 0, 1.0, False),        # fewer than 64 kept rows of a wide layer
])
def test_backward_on_cuda_cores(dtype, B, H, W, C_in, C_out, mask, r, accumulate):
    M = B * H * W
    X, Wt, dY = synth.layer_inputs(dtype, M, C_in, C_out, 61)
    keep, _ = oracle.sample_keep(mask, B, H, W, r, 4)
    cap = B * sbp.sbp_keep_count(mask, H, W, r)
    rows = np.zeros(cap, dtype=np.int32)
    rows[:len(keep)] = keep
    rows_d = torch.from_numpy(rows).cuda()
    cnt = torch.tensor([len(keep)], dtype=torch.int32, device="cuda")
    Xk = run_forward_cache(dtype, dev(X, dtype), rows_d, cap, cnt)
    want = oracle.linear_backward(synth.to_f64(X[keep], dtype), synth.to_f64(dY, dtype), synth.to_f64(Wt, dtype), keep)
    init = None
    if accumulate:
        init = dict(dW=torch.linspace(-1, 1, C_in * C_out).reshape(C_in, C_out), db=torch.linspace(2, 3, C_out))
    got = run_backward(dtype, Xk, dev(dY, dtype), dev(Wt, dtype), rows_d, cap, cnt, init=init,
                       flags=(sbp.SBP_FLAG_ACCUMULATE if accumulate else 0) | (sbp.SBP_FLAG_PLAIN_FMA if dtype == "bf16" else 0))
    assert got["status"] == 0
    add = {k: (v.numpy().astype(np.float64) if accumulate else 0.0) for k, v in (init or dict(dW=None, db=None)).items()}
    _check(got["dW"], want["dW"] + add["dW"], dtype, False)
    _check(got["db"], want["db"] + add["db"], dtype, False)
    _check(got["dX"], want["dX"], dtype, True)
    dropped = np.setdiff1d(np.arange(M), keep)
    assert not host(got["dX"])[dropped].view(np.uint8).any()


@pytest.mark.parametrize("dtype,M,C_in,C_out,w_out_in", [
    ("f32", 1, 4, 4, False), ("f32", 65, 20, 132, True), ("f32", 63, 64, 60, False), ("f32", 2500, 36, 1028, False),
    ("f32", 2500, 36, 1028, True), ("bf16", 127, 72, 136, False), ("bf16", 64, 8, 64, True),
])
def test_forward_on_cuda_cores(dtype, M, C_in, C_out, w_out_in):
    X, Wt, _ = synth.layer_inputs(dtype, M, C_in, C_out, 62)
    bias = np.linspace(-1, 1, C_out, dtype=np.float32)
    want = oracle.linear_forward(synth.to_f64(X, dtype), synth.to_f64(Wt, dtype), bias)
    Y = torch.full((M, C_out), float("nan"), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")
    W_d = dev(np.ascontiguousarray(Wt.T) if w_out_in else Wt, dtype)
    sbp.sbp_linear_forward(dt_code(dtype), dev(X, dtype), W_d, torch.from_numpy(bias).cuda(), M, C_in, C_out, Y,
                           flags=sbp.SBP_FLAG_PLAIN_FMA | (sbp.SBP_FLAG_W_OUT_IN if w_out_in else 0))
    torch.cuda.synchronize()
    _check(Y, want, dtype, True)


@pytest.mark.parametrize("M,kept,valid,C_in,C_out,out_in", [
    (1176, 294, 294, 68, 260, False), (1400, 700, 700, 1028, 1540, False), (1400, 700, 651, 1028, 1540, True),      # 64 x 128 tiles
    (40000, 20000, 19990, 36, 68, False),                                                                          # the same, long and thin
    (3000, 1500, 1500, 768, 100, True),
])
def test_fp32_backward_on_the_cuda_cores_by_request(M, kept, valid, C_in, C_out, out_in):
    """Sizes that the tensor-core kernel takes by default: SBP_FLAG_PLAIN_FMA keeps them here."""
    X, Wt, dY = synth.layer_inputs("f32", M, C_in, C_out, 63)
    keep = np.sort(np.random.default_rng(9).permutation(M)[:kept]).astype(np.int32)
    rows, count = torch.from_numpy(keep).cuda(), torch.tensor([valid], dtype=torch.int32, device="cuda")
    want = oracle.linear_backward(synth.to_f64(X[keep[:valid]], "f32"), synth.to_f64(dY, "f32"), synth.to_f64(Wt, "f32"), keep[:valid])
    W = dev(np.ascontiguousarray(Wt.T) if out_in else Wt, "f32")
    nb = sbp.sbp_linear_backward_workspace_bytes(sbp.SBP_F32, M, kept, C_in, C_out)
    ws, st = torch.empty(nb, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    dW, db, dX = torch.full_like(W, float("nan")), torch.full((C_out,), float("nan"), device="cuda"), torch.full((M, C_in), float("nan"), device="cuda")
    sbp.sbp_linear_backward(sbp.SBP_F32, dev(X[keep], "f32"), dev(dY, "f32"), W, rows, count, M, kept, C_in, C_out, dW, db, dX,
                            sbp.SBP_FLAG_PLAIN_FMA | (sbp.SBP_FLAG_W_OUT_IN if out_in else 0), ws, nb, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    _check(dW.t().contiguous() if out_in else dW, want["dW"], "f32", False)
    _check(db, want["db"], "f32", False)
    _check(dX, want["dX"], "f32", True)
    assert not host(dX)[np.setdiff1d(np.arange(M), keep[:valid])].view(np.uint8).any()
