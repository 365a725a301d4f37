"""Overflowed gradients (a loss scale that was too large) stay visible: infinities, NaNs and sums beyond the range of fp32 arrive in
db as they would from plain additions - an infinity does not become a NaN, and neighbouring columns are untouched."""
import numpy as np
import pytest
import torch

import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, dt_code, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,M_keep,C_in,C_out,flags", [
    ("f32", 40, 36, 68, 0), ("f32", 2000, 64, 64, 0), ("f32", 700, 768, 772, 0), ("f32", 300, 128, 132, 64), ("f32", 2000, 2048, 260, 64),
    ("bf16", 200, 72, 40, 8), ("bf16", 600, 96, 96, 0), ("bf16", 3000, 512, 640, 0),
])
def test_bias_gradient_of_infinite_columns(dtype, M_keep, C_in, C_out, flags):
    M = 2 * M_keep
    X, W, dY = synth.layer_inputs(dtype, M_keep, C_in, C_out, 71)
    rows = (np.arange(M_keep) * 2 + 1).astype(np.int32)
    full = np.zeros((M, C_out), dtype=np.float32)
    full[rows] = synth.to_f64(dY, dtype)
    big = np.float32(2.0 ** 127)
    full[rows[7], 1] = np.inf
    full[rows[M_keep // 2], 2] = -np.inf
    full[rows[-1], 3] = np.nan
    full[rows[3], 4], full[rows[-2], 4] = np.inf, -np.inf
    full[rows[[0, 5, 20]], 5] = big                      # 3 x 2^127 is beyond fp32
    full[rows[[1, -1]], C_out - 1] = -big
    t = torch.from_numpy(full).cuda()
    dY_d = t.to(torch.bfloat16) if dtype == "bf16" else t
    W_d = dev(np.ascontiguousarray(W.T) if flags & sbp.SBP_FLAG_W_OUT_IN else W, dtype)
    code = dt_code(dtype)
    nb = sbp.sbp_linear_backward_workspace_bytes(code, M, M_keep, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    dW = torch.empty(tuple(W_d.shape), device="cuda")
    db = torch.empty(C_out, device="cuda")
    dX = torch.empty(M, C_in, dtype=dY_d.dtype, device="cuda")
    sbp.sbp_linear_backward(code, dev(X, dtype), dY_d, W_d, torch.from_numpy(rows).cuda(), None, M, M_keep, C_in, C_out, dW, db, dX, flags, ws, nb)
    torch.cuda.synchronize()
    got = host(db).astype(np.float64)
    exact = host(dY_d.double())[rows].sum(0)
    with np.errstate(over="ignore"):
        want = exact.astype(np.float32)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
    ok = np.isfinite(want)
    assert ok.sum() == C_out - 6
    # fp32 sums of M_keep terms
    assert np.abs(got[ok] - exact[ok]).max() <= 1e-5 * np.sqrt(M_keep) * np.abs(host(dY_d.double())[rows][:, ok]).max()
