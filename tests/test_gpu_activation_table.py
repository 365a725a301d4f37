"""`sbp_act_backward` on bf16 arrays large enough for the tabulated derivative: every bf16 bit pattern as Z (both ends of
the table, both signs, subnormals, infinities, NaNs), one vector below the smallest such array, at it, and above it."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, host

pytestmark = pytest.mark.gpu
TABLE_FROM = 148 * 4 * 1024          # 16-byte vectors


@pytest.mark.parametrize("vectors,padding", [(TABLE_FROM - 1, 0), (TABLE_FROM, 0), (TABLE_FROM + 777, 1234)])
def test_gelu_derivative_at_every_bf16_number(vectors, padding):
    n = vectors * 8
    bits = (np.arange(n, dtype=np.uint32) & 0xFFFF).astype(np.uint16)
    dH = np.full(n, synth.f64_to_bf16_bits(np.array([3.0]))[0], dtype=np.uint16)
    cnt = torch.tensor([vectors - padding], dtype=torch.int32, device="cuda")
    out = torch.full((vectors, 8), 7.0, dtype=torch.bfloat16, device="cuda")
    sbp.sbp_act_backward(sbp.SBP_BF16, sbp.SBP_ACT_GELU, dev(bits.reshape(-1, 8), "bf16"), dev(dH.reshape(-1, 8), "bf16"), cnt, vectors, 8, out)
    torch.cuda.synchronize()
    got_bits = host(out).reshape(-1)
    live = n - padding * 8
    assert not got_bits[live:].any()                                          # padding rows: +0.0
    assert live > 2 * 65536
    got = got_bits[:live]
    assert (got[65536:] == got[np.arange(65536, live) & 0xFFFF]).all()        # the same number, the same answer everywhere
    z = synth.bf16_bits_to_f64(bits[:65536])
    with np.errstate(over="ignore", invalid="ignore"):
        finite = np.isfinite(z) & (np.abs(z) < 1e18)                          # beyond: z * z overflows fp32 (exp gives 0 all the same)
    want = oracle.act_backward_gelu(z[finite].reshape(1, -1), np.full((1, int(finite.sum())), 3.0)).reshape(-1)
    err = np.abs(synth.bf16_bits_to_f64(got[:65536])[finite] - want)
    # one rounding to bf16 (8 significant bits: at most 2^-8 of the value) beside fp32 erff and expf, whose absolute error near the zero of gelu' and in
    # its tail is a few 2^-24 of the terms (at most 3 * 1.2)
    assert (err <= 2.0 ** -8 * np.abs(want) + 2e-6).all()
    assert np.isnan(synth.bf16_bits_to_f64(got[:65536])[np.isnan(z)]).all()
