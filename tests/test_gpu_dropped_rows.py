"""Zero rows of dX from the tensor-core kernel, cleared in equal shares of its rows: gaps longer and shorter than a share, kept
rows only at the start, only at the end, in whole frames, none at all, and the padding rows of a packed dX."""
import numpy as np
import pytest
import torch

import paper_2210_00129_b200 as sbp
from gpu_harness import run_backward

pytestmark = pytest.mark.gpu

LISTS = {
    "start": lambda M, n: np.arange(n),
    "end": lambda M, n: np.arange(M - n, M),
    "frames": lambda M, n: np.concatenate([np.arange(f * 196, f * 196 + 196) for f in range(1, M // 196, 2)])[:n],
    "every other": lambda M, n: np.arange(1, M, 2)[:n],
    "one": lambda M, n: np.array([M // 2]),
    "none": lambda M, n: np.array([], dtype=np.int64),
}


@pytest.mark.parametrize("kind", list(LISTS))
@pytest.mark.parametrize("M,C_in,C_out,packed", [(1568, 768, 256, False), (4001, 136, 512, False), (9600, 520, 264, False), (9600, 520, 264, True)])
def test_dropped_rows_are_zero(kind, M, C_in, C_out, packed):
    cap = M // 2
    keep = LISTS[kind](M, cap)
    n = len(keep)
    rows = torch.zeros(cap, dtype=torch.int32)
    rows[:n] = torch.from_numpy(keep).int()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M)
    dY = torch.randn(M, C_out, device="cuda", generator=gen).bfloat16()
    W = (torch.randn(C_in, C_out, device="cuda", generator=gen) * 0.02).bfloat16()
    Xk = torch.zeros(cap, C_in, device="cuda", dtype=torch.bfloat16)
    Xk[:n] = torch.randn(n, C_in, device="cuda", generator=gen).bfloat16()
    cnt = torch.tensor([n], dtype=torch.int32, device="cuda")
    got = run_backward("bf16", Xk, dY, W, rows.cuda(), cap, cnt, flags=sbp.SBP_FLAG_DX_COMPACT if packed else 0, dX_rows=cap if packed else None)
    assert got["status"] == 0
    at = torch.arange(n, device="cuda") if packed else torch.from_numpy(keep).cuda()
    want = dY[torch.from_numpy(keep).cuda()].double() @ W.double().t()
    dropped = torch.ones(got["dX"].shape[0], dtype=torch.bool, device="cuda")
    dropped[at] = False
    assert not got["dX"][dropped].view(torch.int16).any()                     # +0.0 bits
    if n:                                                                     # one rounding to bf16 beside fp32 sums
        err = (got["dX"][at].double() - want).abs()
        assert bool((err <= 2.0 ** -8 * want.abs() + 1e-4 * want.pow(2).mean().sqrt()).all())
    want_dW = Xk[:n].double().t() @ dY[torch.from_numpy(keep).cuda()].double()
    assert bool((got["dW"].double() - want_dW).abs().max() <= 1e-3 * max(float(want_dW.pow(2).mean().sqrt()), 1e-30) if n else not got["dW"].any())
