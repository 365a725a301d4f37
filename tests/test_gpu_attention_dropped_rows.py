"""`sbp_attention_backward` with more problems than resident blocks (296, or 148 with more than 128 tokens a side), where each warp clears a
share of the rows that the lists leave out, or each problem its own: every documented pair of subsets, fused and separate layouts, shares
that are equal, uneven and empty, ragged lists with empty samples, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, host

pytestmark = pytest.mark.gpu
D = 64


def _lists(rng, B, N, most):
    counts = [most if b == 0 else 0 if b % 11 == 5 else int(rng.integers(1, most + 1)) for b in range(B)]
    rows = np.concatenate([b * N + np.sort(rng.permutation(N)[:n]) for b, n in enumerate(counts)])
    return rows.astype(np.int32), np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)


def _call(B, N, heads, kind, fused, tensors, lists, most, flags=0):
    """Outputs [3][B * N, heads * 64] (NaN before the call) of Q, K, V, dA."""
    M, C = B * N, heads * D
    if fused:
        qkv, out = dev(np.concatenate(tensors[:3], axis=1), "bf16"), torch.full((M, 3 * C), float("nan"), dtype=torch.bfloat16, device="cuda")
        (q, k, v), grads, ld = [qkv[:, i * C:] for i in range(3)], [out[:, i * C:] for i in range(3)], 3 * C
    else:
        q, k, v = (dev(a, "bf16") for a in tensors[:3])
        grads, ld = [torch.full((M, C), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3)], C
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    (qr, qo), (kr, ko) = ((None, None) if l is None else tuple(torch.from_numpy(a).cuda() for a in l) for l in lists)
    flags |= sbp.SBP_FLAG_ATTN_ALL_KEYS if kind == "query" else 0
    sbp.sbp_attention_backward(sbp.SBP_BF16, q, k, v, ld, dev(tensors[3], "bf16"), C, qr, qo, kr, ko, B, N, heads, D, most, *grads, ld, flags, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    return [host(g[:, :C].contiguous()) for g in grads]


@pytest.mark.parametrize("B,N,heads,most,kind,fused", [
    (75, 40, 4, 20, "qkv", True),          # a few problems more than blocks
    (37, 33, 16, 17, "qkv", True),         # as many for each block: each problem its own rows
    (48, 60, 12, 30, "qkv", False),        # all but a few blocks have two
    (310, 21, 1, 8, "qkv", True), (160, 40, 2, 20, "qkv", False), (102, 30, 3, 9, "qkv", False),        # few heads: several rows at a time
    (60, 100, 5, 9, "keys", True),         # every token a query, listed keys
    (50, 128, 6, 64, "query", True), (200, 17, 3, 8, "two", False),
    (230, 256, 2, 64, "qkv", True),        # shares for the blocks with two problems, larger ones for the others
    # one block an SM
    (40, 200, 4, 98, "query", True), (74, 140, 4, 70, "query", False), (50, 180, 3, 150, "qkv", True), (20, 256, 8, 129, "keys", False),
    (155, 150, 1, 140, "two", True), (36, 240, 8, 60, "query", False), (34, 240, 8, 60, "query", True),
])
def test_rows_outside_the_lists(B, N, heads, most, kind, fused):
    rng = np.random.default_rng(B * heads + N)
    M, C = B * N, heads * D
    tensors = [synth.gaussian_tensor((M, C), "bf16", 900 + N, i, 1.0 if i < 3 else 1e-2) for i in range(4)]
    listed, everything = _lists(rng, B, N, most), (np.arange(M, dtype=np.int32), np.arange(0, M + 1, N, dtype=np.int32))
    q_list, k_list = {"qkv": (listed, listed), "query": (listed, everything), "keys": (everything, listed), "two": (listed, _lists(rng, B, N, most))}[kind]
    given = {"qkv": (listed, None), "query": (listed, None), "keys": (None, listed), "two": (q_list, k_list)}[kind]
    got = _call(B, N, heads, kind, fused, tensors, given, most)
    f = synth.bf16_bits_to_f64
    want = oracle.attention_backward(*(f(a) for a in tensors), *q_list, *k_list, heads)
    for name, bits, w, (rows, _) in zip(("dQ", "dK", "dV"), got, want, (q_list, k_list, k_list)):
        dropped = np.setdiff1d(np.arange(M), rows)
        assert not bits[dropped].any(), name
        # S and dM are rounded to bf16 between the products (2^-9 of each term, random in sign), the result once more
        assert np.linalg.norm(f(bits) - w) <= 5e-3 * np.linalg.norm(w) + 1e-12, name
