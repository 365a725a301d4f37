"""SBP_FLAG_W_OUT_IN on weights large enough to be read and written in place: every tile shape of the kernels (narrow, wide,
pairs of blocks, role split, CUDA cores), ragged edges, accumulation, split reductions and the packed forms, against the
oracle or - at sizes the oracle is slow on - the [C_in, C_out] layout of the same call."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, dt_code, host

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "bf16": 5e-3}


def _call(dtype, Xk, dY, W, rows, cnt, M, cap, ci, co, flags, dW0=None, db0=None, dX_rows=None):
    code = dt_code(dtype)
    nb = sbp.sbp_linear_backward_workspace_bytes(code, M, cap, ci, co)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    dW = dW0.clone() if dW0 is not None else torch.full(tuple(W.shape), float("nan"), device="cuda")
    db = db0.clone() if db0 is not None else torch.full((co,), float("nan"), device="cuda")
    dX = torch.full((M if dX_rows is None else dX_rows, ci), float("nan"), dtype=W.dtype, device="cuda")
    sbp.sbp_linear_backward(code, Xk, dY, W, rows, cnt, M, cap, ci, co, dW, db, dX, flags, ws, nb, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    return dW, db, dX


@pytest.mark.parametrize("dtype,B,H,W,C_in,C_out,accumulate", [
    ("bf16", 5, 14, 14, 512, 384, False),
    ("bf16", 3, 14, 14, 520, 264, True),        # ragged tiles in both directions
    ("bf16", 4, 28, 28, 136, 1032, True),       # 128-wide tiles, db out of the dW tiles
    ("bf16", 3, 15, 13, 1032, 136, False),
    ("f32", 3, 13, 11, 260, 516, True),
])
def test_in_place_layout_matches_the_oracle(dtype, B, H, W, C_in, C_out, accumulate):
    M = B * H * W
    assert C_in * C_out >= 1 << 17
    X, Wt, dY = synth.layer_inputs(dtype, M, C_in, C_out, 81)
    keep, _ = oracle.sample_keep(0, B, H, W, 0.5, 2)
    n = len(keep)
    want = oracle.linear_backward(synth.to_f64(X[keep], dtype), synth.to_f64(dY, dtype), synth.to_f64(Wt, dtype), keep)
    dW0 = torch.linspace(-1, 1, C_in * C_out, device="cuda").reshape(C_out, C_in) if accumulate else None
    db0 = torch.linspace(2, 3, C_out, device="cuda") if accumulate else None
    flags = sbp.SBP_FLAG_W_OUT_IN | (sbp.SBP_FLAG_ACCUMULATE if accumulate else 0)
    dW, db, dX = _call(dtype, dev(X[keep], dtype), dev(dY, dtype), dev(np.ascontiguousarray(Wt.T), dtype), torch.from_numpy(keep).cuda(), None,
                       M, n, C_in, C_out, flags, dW0, db0)
    rms = lambda a: float(np.sqrt(np.mean(a * a)))
    for got, w, base in ((dW, want["dW"].T, dW0), (db, want["db"], db0)):
        g = host(got).astype(np.float64) - (host(base).astype(np.float64) if accumulate else 0.0)
        # fp32 sums of n terms of either sign, added to starting values of up to 3: a few times 2^-24 of those beside 1e-4 rms
        assert np.abs(g - w).max() <= (1e-4 if dtype == "f32" else 1e-3) * rms(w) + (1e-6 if accumulate else 0.0)
    dX_bits = host(dX)
    assert np.linalg.norm(synth.to_f64(dX_bits, dtype) - want["dX"]) <= TOL[dtype] * np.linalg.norm(want["dX"])
    assert not dX_bits[np.setdiff1d(np.arange(M), keep)].view(np.uint8).any()


@pytest.mark.parametrize("M,ci,co,mask,flags", [
    (9200, 776, 520, 0, 0),                                            # pairs of blocks, odd tile counts
    (9200, 1032, 264, 0, sbp.SBP_FLAG_ACCUMULATE),
    (9200, 512, 776, 0, sbp.SBP_FLAG_DX_COMPACT),
    (9200, 512, 776, 0, sbp.SBP_FLAG_DY_COMPACT),
    (300000, 1024, 128, 0, 0),                                         # memory-bound: role split
    (64 * 49, 1024, 4096, 1, 0),                                       # count on the device, split reduction
])
def test_in_place_layout_equals_the_other_one(M, ci, co, mask, flags):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    rn = lambda *s: torch.randn(*s, device="cuda", generator=gen)
    if mask:
        cap = 64 * sbp.sbp_keep_count(1, 7, 7, 0.5)
        rows, offs = torch.zeros(cap, dtype=torch.int32, device="cuda"), torch.zeros(65, dtype=torch.int32, device="cuda")
        sbp.sbp_sample_keep(1, 64, 7, 7, 0.5, 1, 2, 0, 0, rows, offs)
        cnt = offs[64:]
    else:
        cap = M // 2
        rows = torch.randperm(M, device="cuda", generator=gen)[:cap].sort().values.int()
        cnt = None
    Xk, W = rn(cap, ci).bfloat16(), (rn(ci, co) * 0.02).bfloat16()
    dY = rn(cap if flags & sbp.SBP_FLAG_DY_COMPACT else M, co).bfloat16()
    acc = bool(flags & sbp.SBP_FLAG_ACCUMULATE)
    dW0, db0 = (rn(ci, co), rn(co)) if acc else (None, None)
    dX_rows = cap if flags & sbp.SBP_FLAG_DX_COMPACT else None
    a = _call("bf16", Xk, dY, W, rows, cnt, M, cap, ci, co, flags, dW0, db0, dX_rows)
    b = _call("bf16", Xk, dY, W.t().contiguous(), rows, cnt, M, cap, ci, co, flags | sbp.SBP_FLAG_W_OUT_IN,
              dW0.t().contiguous() if acc else None, db0, dX_rows)
    # the same products in the same order: only the layout differs
    assert torch.equal(a[0], b[0].t()) and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
