"""bf16 layers with a side below 128 channels, or few rows, on the tensor cores: down to 8 channels and one kept row, both sides
of the lines to the CUDA cores, both weight layouts, accumulation and device-side counts, against the product in 64 bits."""
import pytest
import torch

import paper_2210_00129_b200 as sbp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap,keep,C_in,C_out,w_out_in,accumulate", [
    (1, 1, 8, 8, False, False), (5, 3, 8, 264, False, True), (63, 63, 264, 8, False, False), (64, 50, 24, 56, False, True),
    (130, 129, 64, 64, False, False), (512, 512, 256, 32, False, False), (513, 500, 256, 32, False, True), (512, 512, 264, 40, False, False),
    (700, 650, 120, 72, False, False), (3000, 2999, 64, 2048, True, True), (3000, 2000, 2056, 64, True, False),
    (5000, 4500, 8, 16384, True, False), (5000, 4500, 16384, 8, True, True), (6000, 5000, 96, 520, False, False), (5000, 5000, 512, 72, False, False),
    (200, 0, 64, 136, False, False), (200, 0, 64, 136, False, True), (784, 700, 768, 768, False, True), (784, 784, 768, 768, True, False),
    (1500, 1400, 2048, 2048, False, False), (1111, 1111, 2056, 1032, False, True), (3000, 2990, 3072, 768, True, False), (3001, 2875, 3080, 264, False, False),  # wide, few rows
    (16000, 15873, 512, 128, False, False), (20000, 19990, 264, 264, False, True), (30000, 28000, 64, 64, True, False),         # dW and dX blocks apart
])
def test_narrow_backward(cap, keep, C_in, C_out, w_out_in, accumulate):
    M = 2 * cap + 3
    gen = torch.Generator(device="cuda")
    gen.manual_seed(cap + C_in)
    rows = torch.zeros(cap, dtype=torch.int32, device="cuda")
    pick = torch.randperm(M, device="cuda", generator=gen)[:keep].sort().values
    rows[:keep] = pick.int()
    cnt = torch.tensor([keep], dtype=torch.int32, device="cuda")
    Xk = torch.zeros(cap, C_in, device="cuda", dtype=torch.bfloat16)
    Xk[:keep] = torch.randn(keep, C_in, device="cuda", generator=gen).bfloat16()
    dY = torch.randn(M, C_out, device="cuda", generator=gen).bfloat16()
    W = (torch.randn(C_in, C_out, device="cuda", generator=gen) * 0.02).bfloat16()
    dW = torch.randn(*(W.t() if w_out_in else W).shape, device="cuda", generator=gen) if accumulate else torch.full(tuple((W.t() if w_out_in else W).shape), float("nan"), device="cuda")
    db = torch.randn(C_out, device="cuda", generator=gen) if accumulate else torch.full((C_out,), float("nan"), device="cuda")
    dW0, db0 = (dW.double(), db.double()) if accumulate else (0.0, 0.0)
    dX = torch.full((M, C_in), float("nan"), device="cuda", dtype=torch.bfloat16)
    nb = sbp.sbp_linear_backward_workspace_bytes(sbp.SBP_BF16, M, cap, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    flags = (sbp.SBP_FLAG_W_OUT_IN if w_out_in else 0) | (sbp.SBP_FLAG_ACCUMULATE if accumulate else 0)
    sbp.sbp_linear_backward(sbp.SBP_BF16, Xk, dY, W.t().contiguous() if w_out_in else W, rows, cnt, M, cap, C_in, C_out, dW, db, dX, flags, ws, nb, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    dYk = dY[pick].double()
    want_W = Xk[:keep].double().t() @ dYk
    rms = lambda t: t.pow(2).mean().sqrt()
    # fp32 sums of up to 5000 terms, which lose up to 2^-24 of the sum so far in each 16-deep step, beside the rounding of what
    # they are added to (values of a few units)
    loose = (keep / 16 + 8) * 2.0 ** -24
    assert bool(((dW.double() - dW0) - (want_W.t() if w_out_in else want_W)).abs().max() <= loose * 8 * rms(want_W) + (2e-6 if accumulate else 0))
    want_b = dYk.sum(0)
    assert bool(((db.double() - db0) - want_b).abs().max() <= loose * 8 * rms(want_b) + 1e-5)
    want_X = dYk @ W.double().t()
    err = (dX[pick].double() - want_X).abs()
    assert bool((err <= 2.0 ** -8 * want_X.abs() + (C_out / 16 * 2.0 ** -24 + 1e-5) * rms(want_X)).all())
    dropped = torch.ones(M, dtype=torch.bool, device="cuda")
    dropped[pick] = False
    assert not dX[dropped].view(torch.int16).any()


@pytest.mark.parametrize("w_out_in", [False, True])
@pytest.mark.parametrize("M,C_in,C_out", [(1, 8, 8), (3, 40, 8), (127, 64, 264), (512, 32, 512), (513, 32, 512), (512, 40, 520), (5000, 8, 2048), (5000, 2048, 8),
                                          (20000, 64, 2048)])
def test_narrow_forward(M, C_in, C_out, w_out_in):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + C_in)
    X = torch.randn(M, C_in, device="cuda", generator=gen).bfloat16()
    W = torch.randn(C_in, C_out, device="cuda", generator=gen).bfloat16()
    bias = torch.randn(C_out, device="cuda", generator=gen)
    Y = torch.full((M, C_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    sbp.sbp_linear_forward(sbp.SBP_BF16, X, W.t().contiguous() if w_out_in else W, bias, M, C_in, C_out, Y,
                           flags=sbp.SBP_FLAG_W_OUT_IN if w_out_in else 0, status_word=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    want = X.double() @ W.double() + bias.double()
    err = (Y.double() - want).abs()
    assert bool((err <= 2.0 ** -8 * want.abs() + (C_in / 16 * 2.0 ** -24 + 1e-5) * want.pow(2).mean().sqrt()).all())
