"""`sbp_attention_backward` where its buffers, tiles and layouts change: token bounds around multiples of 16, 64 and 128 on
either side, ragged lists (an empty sample among them), more problems than resident blocks, against the fp64 oracle."""
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
    rows, offs = [], [0]
    for b in range(B):
        n = most if b == 0 else 0 if b == empty else int(rng.integers(1, most + 1))
        rows.append(b * N + np.sort(rng.permutation(N)[:n]))
        offs.append(offs[-1] + n)
    return np.concatenate(rows).astype(np.int32), np.array(offs, dtype=np.int32)


@pytest.mark.parametrize("B,N,heads,q_most,k_most", [
    (3, 5, 1, 1, 1), (3, 40, 2, 16, 17), (3, 70, 2, 64, 65), (3, 130, 2, 48, 112), (3, 130, 1, 112, 113), (3, 200, 1, 128, 128),
    (3, 200, 1, 128, 129), (3, 200, 1, 129, 64), (3, 200, 1, 98, 193), (3, 256, 1, 130, 1), (3, 256, 1, 200, 256), (3, 256, 1, 256, 256),
    (60, 20, 6, 9, 11), (40, 132, 4, 130, 130),
])
def test_attention_at_tile_edges(B, N, heads, q_most, k_most):
    rng = np.random.default_rng(q_most * 1000 + k_most)
    M, C = B * N, heads * D
    Q, K, V, dA = (synth.gaussian_tensor((M, C), "bf16", 300 + q_most, i, 1.0 if i < 3 else 1e-2) for i in range(4))
    empty = 1 if B > 2 else -1
    qr, qo = _lists(rng, B, N, q_most, empty)
    kr, ko = _lists(rng, B, N, k_most, empty)
    out = [torch.full((M, C), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    t = lambda a: torch.from_numpy(a).cuda()
    sbp.sbp_attention_backward(sbp.SBP_BF16, dev(Q, "bf16"), dev(K, "bf16"), dev(V, "bf16"), C, dev(dA, "bf16"), C, t(qr), t(qo), t(kr), t(ko),
                               B, N, heads, D, max(q_most, k_most), *out, C, 0, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    f = synth.bf16_bits_to_f64
    want = oracle.attention_backward(f(Q), f(K), f(V), f(dA), qr, qo, kr, ko, heads)
    for name, g, w, rows in zip(("dQ", "dK", "dV"), out, want, (qr, kr, kr)):
        bits = host(g)
        got = f(bits)
        dropped = np.setdiff1d(np.arange(M), rows)
        assert not bits[dropped].any(), name
        # S and dM are rounded to bf16 between the products: 2^-8 of each term, random in sign, beside the output's own rounding
        rms = float(np.sqrt(np.mean(w[rows] ** 2)))
        assert np.linalg.norm(got - w) <= 5e-3 * np.linalg.norm(w) + 1e-12, name
        assert (np.abs(got - w) <= 2.0 ** -7 * np.abs(w) + 3e-2 * rms + 1e-9).all(), name
