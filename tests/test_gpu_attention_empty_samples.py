"""`sbp_attention_backward` where samples without listed tokens lie between others and every resident block works through
three problems or more: a block's second and later problems are empty, one in a row and several, in both block shapes (up to
128 tokens a side: two blocks an SM, 296 in all; more: one, 148), against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, host

pytestmark = pytest.mark.gpu
D = 64


def _lists(rng, B, N, most, empty):
    counts = [0 if empty(b) else most if b == 0 else int(rng.integers(1, most + 1)) for b in range(B)]
    rows = np.concatenate([b * N + np.sort(rng.permutation(N)[:n]) for b, n in enumerate(counts)])
    return rows.astype(np.int32), np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)


# problems = samples x heads; block i takes problems i, i + blocks, i + 2 blocks, ...
@pytest.mark.parametrize("kept_only", [False, True])
@pytest.mark.parametrize("B,N,heads,q_most,k_most,resident,empty", [
    (960, 24, 1, 17, 16, 296, "second"),        # every block: full, empty, full, full
    (1200, 24, 1, 16, 9, 296, "middle"),        # full, empty, empty, full, full
    (480, 150, 1, 20, 130, 148, "second"),
    (600, 150, 1, 130, 140, 148, "middle"),
    (320, 150, 2, 129, 12, 148, "second"),
])
def test_empty_samples_between_others(B, N, heads, q_most, k_most, resident, empty, kept_only):
    rng = np.random.default_rng(B + q_most)
    M, C = B * N, heads * D
    Q, K, V, dA = (synth.gaussian_tensor((M, C), "bf16", 700 + q_most, i, 1.0 if i < 3 else 1e-2) for i in range(4))
    last = 3 if empty == "middle" else 2
    is_empty = lambda b: resident <= b * heads < last * resident
    qr, qo = _lists(rng, B, N, q_most, is_empty)
    kr, ko = _lists(rng, B, N, k_most, is_empty)
    assert B * heads > 3 * resident
    f = synth.bf16_bits_to_f64
    want = oracle.attention_backward(f(Q), f(K), f(V), f(dA), qr, qo, kr, ko, heads)
    t = lambda a: torch.from_numpy(a).cuda()
    args = [dev(a, "bf16") for a in (Q, K, V, dA)] + [t(a) for a in (qr, qo, kr, ko)]
    for _ in range(3):
        out = [torch.full((M, C), -7.0, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        sbp.sbp_attention_backward(sbp.SBP_BF16, args[0], args[1], args[2], C, args[3], C, *args[4:], B, N, heads, D,
                                   max(q_most, k_most), *out, C, sbp.SBP_FLAG_ATTN_KEPT_ROWS_ONLY if kept_only else 0, st)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        for name, g, w, rows in zip(("dQ", "dK", "dV"), out, want, (qr, kr, kr)):
            bits = host(g)
            got = f(bits)
            other = np.setdiff1d(np.arange(M), rows)
            assert (got[other] == -7.0).all() if kept_only else not bits[other].any(), name
            # S and dM are rounded to bf16 between the products: 2^-9 of each term, random in sign, so that an element is off by some
            # 2^-9 of its row's root mean square (fifteen times that is allowed: there are a million elements), beside the output's
            # own rounding; rows whose terms cancel are held to a thousandth of the whole
            w, got = w[rows], got[rows]
            assert np.linalg.norm(got - w) <= 5e-3 * np.linalg.norm(w) + 1e-12, name
            row_rms = np.sqrt(np.mean(w.reshape(len(rows), heads, D) ** 2, axis=2)).repeat(D, axis=1)
            assert (np.abs(got - w) <= 2.0 ** -8 * np.abs(w) + 3e-2 * row_rms + 1e-3 * np.sqrt(np.mean(w ** 2))).all(), name


@pytest.mark.parametrize("kept_only", [False, True])
@pytest.mark.parametrize("B,N,heads,q_most,k_most,all_keys,empty_side", [
    (5, 40, 2, 33, 20, False, "q"), (5, 40, 2, 33, 20, False, "k"), (400, 20, 1, 9, 16, False, "q"), (400, 20, 1, 9, 16, False, "k"),
    (4, 200, 2, 20, 190, False, "q"), (4, 200, 1, 190, 20, False, "k"), (3, 60, 2, 30, 60, True, "q"), (3, 150, 1, 30, 150, True, "q"),
])
def test_samples_with_one_side_empty(B, N, heads, q_most, k_most, all_keys, empty_side, kept_only):
    """Queries without keys, keys without queries: the gradients of the listed tokens are sums over nothing, +0.0."""
    rng = np.random.default_rng(B + N)
    M, C = B * N, heads * D
    Q, K, V, dA = (synth.gaussian_tensor((M, C), "bf16", 800 + N, i, 1.0 if i < 3 else 1e-2) for i in range(4))
    odd = lambda b: b % 2 == 1
    never = lambda b: False
    qr, qo = _lists(rng, B, N, q_most, odd if empty_side == "q" else never)
    kr, ko = _lists(rng, B, N, k_most, odd if empty_side == "k" else never)
    if all_keys:
        kr, ko = np.arange(M, dtype=np.int32), np.arange(0, M + 1, N, dtype=np.int32)
    t = lambda a: torch.from_numpy(a).cuda()
    out = [torch.full((M, C), -7.0, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    flags = (sbp.SBP_FLAG_ATTN_KEPT_ROWS_ONLY if kept_only else 0) | (sbp.SBP_FLAG_ATTN_ALL_KEYS if all_keys else 0)
    k_args = (None, None) if all_keys else (t(kr), t(ko))
    sbp.sbp_attention_backward(sbp.SBP_BF16, *(dev(a, "bf16") for a in (Q, K, V)), C, dev(dA, "bf16"), C, t(qr), t(qo), *k_args, B, N,
                               heads, D, max(q_most, 0 if all_keys else k_most), *out, C, flags)
    torch.cuda.synchronize()
    listed_q, listed_k = np.zeros(M, dtype=bool), np.zeros(M, dtype=bool)
    listed_q[qr], listed_k[kr] = True, True
    one_sided = (np.arange(M) // N) % 2 == 1
    for name, g, listed in zip(("dQ", "dK", "dV"), out, (listed_q, listed_k, listed_k)):
        bits = host(g)
        assert not bits[listed & one_sided].any(), name
        assert bits[listed & ~one_sided].any(), name
        if kept_only:
            assert (synth.bf16_bits_to_f64(bits[~listed]) == -7.0).all(), name
        else:
            assert not bits[~listed].any(), name
