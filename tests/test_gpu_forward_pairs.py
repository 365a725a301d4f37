"""sbp_linear_forward on 256-wide tiles shared by pairs of blocks: one tile, a dead second half, ragged rows, columns and
depth, more tiles than pairs, both weight layouts, with and without the cache, against the same product in 64 bits."""
import pytest
import torch

import paper_2210_00129_b200 as sbp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w_out_in", [False, True])
@pytest.mark.parametrize("M,C_in,C_out,cap", [
    (128, 128, 256, 0), (300, 520, 776, 0),                     # single blocks
    (128, 12800, 2304, 0),                                      # one row of tiles, their second halves dead
    (129, 12808, 2312, 0), (2000, 3848, 520, 1000),             # ragged rows, columns and depth
    (40000, 264, 264, 9000), (5000, 768, 2304, 2500),           # more tiles than pairs
])
def test_forward_in_pairs(M, C_in, C_out, cap, w_out_in):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + C_out)
    X = torch.randn(M, C_in, device="cuda", generator=gen).bfloat16()
    W = (torch.randn(C_in, C_out, device="cuda", generator=gen) * 0.02).bfloat16()
    bias = torch.randn(C_out, device="cuda", generator=gen)
    Y = torch.full((M, C_out), float("nan"), device="cuda", dtype=torch.bfloat16)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    rows = torch.randperm(M, device="cuda", generator=gen)[:cap].sort().values.int() if cap else None
    Xk = torch.full((cap, C_in), float("nan"), device="cuda", dtype=torch.bfloat16) if cap else None
    sbp.sbp_linear_forward(sbp.SBP_BF16, X, W.t().contiguous() if w_out_in else W, bias, M, C_in, C_out, Y, rows, None, cap, Xk,
                           sbp.SBP_FLAG_W_OUT_IN if w_out_in else 0, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    want = X.double() @ W.double() + bias.double()
    # one rounding to bf16, beside C_in / 16 accumulation steps in fp32 which each lose up to 2^-24 of the sum so far
    err = (Y.double() - want).abs()
    assert bool((err <= 2.0 ** -8 * want.abs() + (C_in / 16 * 2.0 ** -24 + 1e-5) * want.pow(2).mean().sqrt()).all())
    if cap:
        assert torch.equal(Xk, X[rows.long()])
