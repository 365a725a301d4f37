"""The copy kernels (forward cache, patch cache, patch scatter) where their spans, cells and slices end: rows of one vector,
rows around a span's length, strides beyond the kernel and beyond the map, cells cut by the map's edges, cells of several
blocks, capacities above the device-side count.  Pure copies: every result is exact."""
import numpy as np
import pytest
import torch

import paper_2210_00129_b200 as sbp

pytestmark = pytest.mark.gpu


def _list(n_rows, n_keep, cap, seed):
    gen = torch.Generator().manual_seed(seed)
    rows = torch.zeros(max(cap, 1), dtype=torch.int32)
    rows[:n_keep] = torch.randperm(n_rows, generator=gen)[:n_keep].sort().values.int()
    return rows.cuda(), torch.tensor([n_keep], dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("M,C,keep,cap", [
    (1, 4, 1, 1), (3000, 4, 1500, 1501), (700, 12, 699, 700), (50, 4 * 1023, 20, 25), (50, 4 * 1024, 20, 20), (50, 4 * 1025, 20, 21),
    (9, 4 * 5000, 4, 9), (40000, 20, 20000, 20003), (64, 260, 0, 7),
])
def test_forward_cache_spans(M, C, keep, cap):
    X = torch.randn(M, C, device="cuda")
    rows, cnt = _list(M, keep, cap, M + C)
    out = torch.full((cap, C), float("nan"), device="cuda")
    sbp.sbp_forward_cache(sbp.SBP_F32, X, M, C, rows, cnt, cap, out)
    torch.cuda.synchronize()
    assert torch.equal(out[:keep], X[rows[:keep].long()])
    assert not out[keep:].view(torch.int32).any()


@pytest.mark.parametrize("B,H,W,C,k,s,ratio", [
    (2, 8, 8, 4, 1, 1, 0.5), (3, 9, 7, 8, 2, 2, 0.5),          # the last row and column belong to no patch
    (2, 14, 11, 4, 2, 5, 0.6), (4, 6, 7, 12, 3, 100, 1.0),      # strides beyond the kernel, beyond the map
    (1, 64, 64, 4, 4, 4, 0.1), (70, 4, 4, 4, 2, 2, 0.5),        # many cells a block; samples inside a block
    (2, 20, 20, 2000, 5, 10, 0.5),                              # a cell is written by many blocks
    (1, 7, 300, 36, 3, 3, 0.0),                                 # nothing kept
])
def test_patch_cache_and_scatter(B, H, W, C, k, s, ratio):
    Ho, Wo = (H - k) // s + 1, (W - k) // s + 1
    Mo, Kc = B * Ho * Wo, k * k * C
    keep = int(round(ratio * Mo))
    cap = min(Mo, keep + 3)
    rows, cnt = _list(Mo, keep, cap, H * W + C)
    X = torch.randn(B, H, W, C, device="cuda")
    Xk = torch.full((cap, Kc), float("nan"), device="cuda")
    sbp.sbp_patch_cache(sbp.SBP_F32, X, B, H, W, C, k, s, rows, cnt, cap, Xk)
    patches = X[:, :(Ho - 1) * s + k, :(Wo - 1) * s + k].unfold(1, k, s).unfold(2, k, s)          # [B, Ho, Wo, C, k, k]
    patches = patches.permute(0, 1, 2, 4, 5, 3).reshape(Mo, Kc)
    pick = rows[:keep].long()
    dXp = torch.randn(cap, Kc, device="cuda")
    nbytes = sbp.sbp_patch_scatter_workspace_bytes(B, H, W, k, s)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    dX = torch.full((B, H, W, C), float("nan"), device="cuda")
    sbp.sbp_patch_scatter(sbp.SBP_F32, dXp, B, H, W, C, k, s, rows, cnt, cap, dX, ws, nbytes)
    torch.cuda.synchronize()
    assert torch.equal(Xk[:keep], patches[pick])
    assert not Xk[keep:].view(torch.int32).any()
    want = torch.zeros(B, H, W, C, device="cuda")
    b, ho, wo = pick // (Ho * Wo), (pick // Wo) % Ho, pick % Wo
    for dh in range(k):
        for dw in range(k):
            want[b, ho * s + dh, wo * s + dw] = dXp[:keep].view(keep, k, k, C)[:, dh, dw]
    assert torch.equal(dX, want)
    assert not (dX.view(torch.int32) == -2147483648).any()                                         # the zeros are +0.0


@pytest.mark.parametrize("order", ["reversed", "shuffled"])
def test_patch_calls_take_rows_in_any_order(order):
    B, H, W, C, k, s = 3, 40, 36, 16, 2, 2
    Mo, Kc, keep = B * (H // k) * (W // k), k * k * C, 500
    gen = torch.Generator().manual_seed(3)
    rows = torch.randperm(Mo, generator=gen)[:keep].int()
    rows = (rows.sort(descending=True).values if order == "reversed" else rows).cuda()
    X = torch.randn(B, H, W, C, device="cuda")
    Xk = torch.empty(keep, Kc, device="cuda")
    sbp.sbp_patch_cache(sbp.SBP_F32, X, B, H, W, C, k, s, rows, None, keep, Xk)
    nbytes = sbp.sbp_patch_scatter_workspace_bytes(B, H, W, k, s)
    dX = torch.full((B, H, W, C), float("nan"), device="cuda")
    # whatever the workspace holds: zeros, ones, valid row numbers of other positions
    for fill in (torch.zeros(nbytes // 4, dtype=torch.int32), torch.full((nbytes // 4,), -1, dtype=torch.int32),
                 torch.arange(nbytes // 4, dtype=torch.int32) % keep):
        ws = fill.cuda()
        sbp.sbp_patch_scatter(sbp.SBP_F32, Xk, B, H, W, C, k, s, rows, None, keep, dX, ws, nbytes)
        torch.cuda.synchronize()
        kept = torch.zeros(Mo, dtype=torch.bool, device="cuda")
        kept[rows.long()] = True
        mask = kept.view(B, H // k, 1, W // k, 1, 1).expand(B, H // k, k, W // k, k, 1).reshape(B, H, W, 1)
        assert torch.equal(dX, torch.where(mask, X, torch.zeros_like(X)))


@pytest.mark.parametrize("H,W,C,k,s,keep", [(72, 72, 2 ** 17, 5, 72, 1), (72, 73, 2 ** 17, 2, 2 ** 31 + 5, 1), (16, 17, 2 ** 23 + 8, 3, 8, 3)])
def test_patch_scatter_with_cells_beyond_a_gigabyte(H, W, C, k, s, keep):
    """Strides far beyond the kernel: every position is a cell of its own (the largest map here takes 4.6 GB)."""
    Ho, Wo = (H - k) // s + 1, (W - k) // s + 1
    assert min(s, H) * min(s, W) * C // 8 > 2 ** 26
    gen = torch.Generator().manual_seed(k)
    rows = torch.randperm(Ho * Wo, generator=gen)[:keep].sort().values.int().cuda()
    dXp = torch.randint(-1000, 1000, (keep, k, k, C), device="cuda", dtype=torch.int16).view(torch.bfloat16)
    dX = torch.full((H, W, C), 3.0, dtype=torch.bfloat16, device="cuda")
    nbytes = sbp.sbp_patch_scatter_workspace_bytes(1, H, W, k, s)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    sbp.sbp_patch_scatter(sbp.SBP_BF16, dXp, 1, H, W, C, k, s, rows, None, keep, dX, ws, nbytes)
    torch.cuda.synchronize()
    bits = dX.view(torch.int16)
    for m, pos in enumerate(rows.tolist()):
        h, w = pos // Wo * s, pos % Wo * s
        patch = bits[h:h + k, w:w + k]
        assert torch.equal(patch, dXp[m].view(torch.int16))
        patch.zero_()
    assert not any(bool(line.any()) for line in bits)              # a row of the map at a time
