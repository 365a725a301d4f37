"""dW over long lists of kept rows on the tensor cores, whose error grows with the length of an accumulation chain: layers with a side
below 128 channels are cut into short pieces, long pieces of the others are summed in parts.  Single blocks, pairs of blocks, dW and
dX blocks apart (with the bias column), cut and uncut tiles, both weight layouts, accumulation, packed gradients."""
import pytest
import torch

import paper_2210_00129_b200 as sbp

pytestmark = pytest.mark.gpu
OI, ACC, PACKED = sbp.SBP_FLAG_W_OUT_IN, sbp.SBP_FLAG_ACCUMULATE, sbp.SBP_FLAG_DY_COMPACT


def longest_chain(M_keep, C_in, C_out):
    """In k-blocks of 64 rows, at most: pieces of 14; otherwise half of the list, where that is more than a piece left whole."""
    return 14 if min(C_in, C_out) < 128 else max(56, (M_keep + 127) // 128)


def rel(got, want):
    return float((got.double() - want).norm() / want.norm())


@pytest.mark.parametrize("M_keep,C_in,C_out,want,flags", [
    (40000, 48, 2048, "wbx", 0), (50176, 16, 1024, "wbx", 0), (50176, 1024, 16, "wb", 0), (30000, 96, 384, "wbx", OI),       # 128-wide tiles
    (25088, 136, 264, "wbx", ACC), (12544, 128, 512, "wbx", 0), (40000, 128, 512, "wbx", 0),
    (66800, 512, 128, "wbx", 0), (50176, 512, 128, "wbx", OI | ACC), (25088, 1024, 256, "wbx", 0), (60001, 256, 64, "wbx", ACC),   # blocks apart
    (25088, 512, 256, "wbx", ACC), (50176, 512, 128, "wbx", PACKED), (30000, 320, 192, "wb", 0), (9000, 320, 192, "w", ACC),       # single wide blocks
    (12544, 768, 2304, "wbx", 0), (25088, 640, 2560, "wbx", OI), (6272, 512, 2048, "wbx", ACC), (20001, 768, 768, "wx", OI | ACC),   # pairs
    (12544, 1000, 1000, "wb", PACKED), (9000, 2048, 2048, "wbx", OI), (1793, 256, 256, "wbx", 0), (2049, 1024, 1024, "wb", 0),      # just past a whole one
])
def test_error_against_the_longest_chain(M_keep, C_in, C_out, want, flags):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M_keep + C_in)
    randn = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)
    M = M_keep + M_keep // 3
    rows = torch.randperm(M, generator=torch.Generator().manual_seed(5))[:M_keep].sort().values.int().cuda()
    Xk, W = randn(M_keep, C_in).bfloat16(), (0.02 * randn(C_in, C_out)).bfloat16()
    dY = randn(M_keep if flags & PACKED else M, C_out).bfloat16()
    kept = (dY if flags & PACKED else dY[rows.long()]).double()
    dW0, db0 = randn(C_out, C_in) if flags & OI else randn(C_in, C_out), randn(C_out)
    dW, db, dX = dW0.clone(), db0.clone(), torch.empty(M, C_in, dtype=torch.bfloat16, device="cuda")
    nb = sbp.sbp_linear_backward_workspace_bytes(1, M, M_keep, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    sbp.sbp_linear_backward(1, Xk, dY, W.t().contiguous() if flags & OI else W, rows, None, M, M_keep, C_in, C_out, dW,
                            db if "b" in want else None, dX if "x" in want else None, flags, ws, nb, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    exact = kept.t() @ Xk.double() if flags & OI else Xk.double().t() @ kept
    # 7e-8 a k-block, and what the parts and pieces add is rounding, below 1e-7
    bound = 7e-8 * longest_chain(M_keep, C_in, C_out) + 1e-7
    assert rel(dW, exact + dW0.double() if flags & ACC else exact) <= bound
    if "b" in want:
        exact = kept.sum(0)
        assert rel(db, exact + db0.double() if flags & ACC else exact) <= 1e-6
    if "x" in want:
        exact = torch.zeros(M, C_in, dtype=torch.double, device="cuda")
        exact[rows.long()] = kept @ W.double().t()
        assert rel(dX, exact) <= 2.0 ** -8 and not dX[(exact == 0).all(1)].view(torch.int16).any()


@pytest.mark.parametrize("count", [0, 1, 64, 20 * 64, 20 * 64 + 1, 30000])
def test_device_side_counts(count):
    """The plan is made for the capacity; how many parts a piece has is known on the device only."""
    for cap, C_in, C_out in ((66800, 512, 128), (66800, 128, 512), (50176, 96, 384), (40000, 768, 768)):
        n = min(count, cap)
        M = cap
        gen = torch.Generator(device="cuda")
        gen.manual_seed(count + C_in)
        Xk = torch.zeros(cap, C_in, dtype=torch.bfloat16, device="cuda")
        Xk[:n] = torch.randn(n, C_in, device="cuda", generator=gen).bfloat16()
        dY = torch.randn(M, C_out, device="cuda", generator=gen).bfloat16()
        W = torch.randn(C_in, C_out, device="cuda", generator=gen).bfloat16()
        rows = torch.arange(cap, dtype=torch.int32, device="cuda")
        rows[:n] = (torch.arange(n, device="cuda") * cap // max(n, 1)).int()
        cnt = torch.tensor([n], dtype=torch.int32, device="cuda")
        dW = torch.full((C_in, C_out), float("nan"), device="cuda")
        db = torch.full((C_out,), float("nan"), device="cuda")
        dX = torch.empty(M, C_in, dtype=torch.bfloat16, device="cuda")
        nb = sbp.sbp_linear_backward_workspace_bytes(1, M, cap, C_in, C_out)
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        sbp.sbp_linear_backward(1, Xk, dY, W, rows, cnt, M, cap, C_in, C_out, dW, db, dX, 0, ws, nb)
        torch.cuda.synchronize()
        kept = dY[rows[:n].long()].double()
        for got, exact in ((dW, Xk[:n].double().t() @ kept), (db, kept.sum(0))):
            assert float((got.double() - exact).norm()) <= (7e-8 * longest_chain(n, C_in, C_out) + 1e-7) * float(exact.norm())
