"""fp32 products on the tensor cores (operands in three bf16 parts) at the edges of their tiles, stages and pieces: against the oracle, and
no further from it than fp32 sums are; infinities and NaNs as the plain products have them."""
import numpy as np
import pytest
import torch

import oracle
import paper_2210_00129_b200 as sbp
from paper_2210_00129_b200 import synth
from gpu_harness import dev, host, run_forward_cache

pytestmark = pytest.mark.gpu

# A stage of 64 is off by at most 4 cuts of 2^-23 of its running sum (a quarter of that on average, and in proportion), the stages add up
# with roundings of 2^-24: sqrt(n / 128) * 2.4e-8 for a depth of n.  1e-7 + 2e-7 up to 8000.
REL = 3e-7


def _rel(got, want):
    return float(np.linalg.norm(host(got).astype(np.float64) - want) / np.linalg.norm(want))


def _elements(got, want):
    scale = float(np.sqrt(np.mean(want * want)))
    return float((np.abs(host(got).astype(np.float64) - want) / np.maximum(np.abs(want), scale)).max())


def _backward(X_keep, dY, W, rows, count, M, cap, C_in, C_out, flags, fill):
    nb = sbp.sbp_linear_backward_workspace_bytes(sbp.SBP_F32, M, cap, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    dW = torch.full_like(W, fill)
    db = torch.full((C_out,), fill, device="cuda")
    dX = torch.full((M, C_in), float("nan"), device="cuda")
    sbp.sbp_linear_backward(sbp.SBP_F32, X_keep, dY, W, rows, count, M, cap, C_in, C_out, dW, db, dX, flags, ws, nb, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return dW, db, dX


@pytest.mark.parametrize("M,kept,padding,C_in,C_out,out_in,accumulate", [
    (1027, 513, 0, 260, 388, False, False),          # one row beyond two row tiles; 4 columns beyond two tiles; depth 4 beyond 6 stages
    (900, 512, 0, 256, 384, False, True),            # full tiles; sums into dW and db
    (1500, 700, 57, 508, 516, True, True),           # rows past the count known on the device; weights [C_out, C_in]
    (6000, 5000, 0, 132, 640, False, False),         # dW cut into pieces
    (4000, 4000, 3000, 384, 132, False, False),      # pieces without rows
    (2000, 1100, 0, 1028, 128, True, False),
    (900, 600, 0, 256, 260, True, True),             # weights [C_out, C_in] small enough to go through transposed copies
])
def test_backward(M, kept, padding, C_in, C_out, out_in, accumulate):
    X, Wt, dY = synth.layer_inputs("f32", M, C_in, C_out, 91)
    keep = np.sort(np.random.default_rng(5).permutation(M)[:kept]).astype(np.int32)
    valid = keep[:kept - padding]
    rows = torch.from_numpy(keep).cuda()
    count = torch.tensor([len(valid)], dtype=torch.int32, device="cuda") if padding else None
    Xk = run_forward_cache("f32", dev(X, "f32"), rows, kept, count)
    want = oracle.linear_backward(synth.to_f64(X[valid], "f32"), synth.to_f64(dY, "f32"), synth.to_f64(Wt, "f32"), valid)
    fill = 0.25 if accumulate else float("nan")
    W = dev(np.ascontiguousarray(Wt.T) if out_in else Wt, "f32")
    flags = (sbp.SBP_FLAG_W_OUT_IN if out_in else 0) | (sbp.SBP_FLAG_ACCUMULATE if accumulate else 0)
    dW, db, dX = _backward(Xk, dev(dY, "f32"), W, rows, count, M, kept, C_in, C_out, flags, fill)
    add = fill if accumulate else 0.0
    for got, exact in ((dW.t() if out_in else dW, want["dW"] + add), (db, want["db"] + add), (dX, want["dX"])):
        assert _rel(got.contiguous(), exact) <= REL and _elements(got.contiguous(), exact) <= 1e-5
    dropped = np.setdiff1d(np.arange(M), valid)
    assert not host(dX)[dropped].view(np.uint8).any()


def test_packed_forms_are_the_scattered_ones():
    """The same numbers, bit for bit, with dY read packed and dX written packed; rows past the count become zeros."""
    M, kept, valid, C_in, C_out = 2000, 1100, 1037, 260, 388
    X, Wt, dY = synth.layer_inputs("f32", M, C_in, C_out, 93)
    rows = torch.from_numpy(np.sort(np.random.default_rng(6).permutation(M)[:kept]).astype(np.int32)).cuda()
    count = torch.tensor([valid], dtype=torch.int32, device="cuda")
    W, dY_d = dev(Wt, "f32"), dev(dY, "f32")
    Xk = run_forward_cache("f32", dev(X, "f32"), rows, kept, count)
    plain = _backward(Xk, dY_d, W, rows, count, M, kept, C_in, C_out, 0, float("nan"))
    packed_dY = dY_d[rows.long()].contiguous()
    from_packed = _backward(Xk, packed_dY, W, rows, count, M, kept, C_in, C_out, sbp.SBP_FLAG_DY_COMPACT, float("nan"))
    both = _backward(Xk, packed_dY, W, rows, count, M, kept, C_in, C_out, sbp.SBP_FLAG_DY_COMPACT | sbp.SBP_FLAG_DX_COMPACT, float("nan"))
    for a, b in zip(plain, from_packed):
        assert torch.equal(a, b)
    assert torch.equal(both[0], plain[0]) and torch.equal(both[1], plain[1])
    assert torch.equal(both[2][:valid], plain[2][rows[:valid].long()]) and not both[2][valid:kept].any()


@pytest.mark.parametrize("M,C_in,C_out,out_in", [(3000, 260, 388, False), (3000, 260, 388, True), (2561, 1028, 900, False), (8192, 512, 128, True)])
def test_forward(M, C_in, C_out, out_in):
    X, Wt, _ = synth.layer_inputs("f32", M, C_in, C_out, 92)
    bias = np.linspace(-1, 1, C_out, dtype=np.float32)
    want = oracle.linear_forward(synth.to_f64(X, "f32"), synth.to_f64(Wt, "f32"), bias)
    Y = torch.full((M, C_out), float("nan"), device="cuda")
    W = dev(np.ascontiguousarray(Wt.T) if out_in else Wt, "f32")
    sbp.sbp_linear_forward(sbp.SBP_F32, dev(X, "f32"), W, torch.from_numpy(bias).cuda(), M, C_in, C_out, Y, flags=sbp.SBP_FLAG_W_OUT_IN if out_in else 0)
    torch.cuda.synchronize()
    assert _rel(Y, want) <= REL and _elements(Y, want) <= 1e-5


@pytest.mark.parametrize("out_in", [False, True])
@pytest.mark.parametrize("accumulate", [False, True])
def test_not_finite(out_in, accumulate):
    """Infinite, NaN and nearly infinite inputs (3.4e38 rounds to infinity in bf16) give what the CUDA-core products give."""
    M, kept, C_in, C_out = 1500, 1100, 512, 384
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    X, dY, W = (torch.randn(*s, device="cuda", generator=g) for s in ((kept, C_in), (M, C_out), (C_out, C_in) if out_in else (C_in, C_out)))
    inf, big = float("inf"), 3.4e38
    rows = torch.arange(0, kept, dtype=torch.int32, device="cuda")
    X[5, 3], X[7, 100], dY[11, 2], dY[12, 5], dY[500, 200] = inf, 1.0, -inf, float("nan"), big
    dY[40] = 0.0
    dY[40, 1] = inf
    W[4, 5], W[8, 9], W[300, 17] = big, inf, -inf
    W[2] = 0.0
    X[:, 20] = 0.0
    X[600, 20] = big
    flags = (sbp.SBP_FLAG_W_OUT_IN if out_in else 0) | (sbp.SBP_FLAG_ACCUMULATE if accumulate else 0)
    run = lambda extra: _backward(X, dY, W, rows, None, M, kept, C_in, C_out, flags | extra, 0.25)
    pairs = list(zip(run(0), run(sbp.SBP_FLAG_PLAIN_FMA)))
    Y = [torch.empty(kept, C_out, device="cuda") for _ in range(2)]
    for y, extra in zip(Y, (0, sbp.SBP_FLAG_PLAIN_FMA)):
        sbp.sbp_linear_forward(sbp.SBP_F32, X, W, None, kept, C_in, C_out, y, flags=(flags & sbp.SBP_FLAG_W_OUT_IN) | extra)
    torch.cuda.synchronize()
    for got, plain in pairs + [tuple(Y)]:
        got, plain = host(got).astype(np.float64), host(plain).astype(np.float64)
        assert np.array_equal(np.isnan(got), np.isnan(plain))
        infinite = np.isinf(plain)
        assert np.array_equal(np.isinf(got), infinite) and np.array_equal(got[infinite], plain[infinite])
        ok = np.isfinite(plain)
        # sums that hold 3.4e38 are compared by themselves: nothing else in them is visible
        assert (np.abs(got[ok] - plain[ok]) <= 1e-5 * np.maximum(np.abs(plain[ok]), 30.0)).all()


@pytest.mark.parametrize("out_in", [False, True])
@pytest.mark.parametrize("x_exp,dy_exp,w_exp", [(0, -118, 0), (-122, 0, 0), (0, 0, -126), (-70, -70, -70), (0, -140, 0), (-140, 12, -140)])
def test_smallest_numbers(x_exp, dy_exp, w_exp, out_in):
    """Operands down to the subnormal numbers keep the bits that an fp32 number has there (parts in bf16 would end at 2^-133)."""
    M, kept, C_in, C_out = 1300, 700, 388, 516
    scale = lambda a, e: (a * np.float32(2.0 ** (e // 2)) * np.float32(2.0 ** (e - e // 2))).astype(np.float32)
    X, Wt, dY = (scale(a, e) for a, e in zip(synth.layer_inputs("f32", M, C_in, C_out, 94), (x_exp, w_exp, dy_exp)))
    keep = np.sort(np.random.default_rng(7).permutation(M)[:kept]).astype(np.int32)
    rows = torch.from_numpy(keep).cuda()
    want = oracle.linear_backward(synth.to_f64(X[keep], "f32"), synth.to_f64(dY, "f32"), synth.to_f64(Wt, "f32"), keep)
    want["Y"] = oracle.linear_forward(synth.to_f64(X, "f32"), synth.to_f64(Wt, "f32"), np.zeros(C_out, dtype=np.float32))
    W = dev(np.ascontiguousarray(Wt.T) if out_in else Wt, "f32")
    flags = sbp.SBP_FLAG_W_OUT_IN if out_in else 0
    dW, db, dX = _backward(dev(X[keep], "f32"), dev(dY, "f32"), W, rows, None, M, kept, C_in, C_out, flags, float("nan"))
    Y = torch.empty(M, C_out, device="cuda")
    sbp.sbp_linear_forward(sbp.SBP_F32, dev(X, "f32"), W, None, M, C_in, C_out, Y, flags=flags)
    torch.cuda.synchronize()
    for name, got in dict(Y=Y, dW=dW.t() if out_in else dW, db=db, dX=dX).items():
        w = want[name]
        off = host(got.contiguous()).astype(np.float64) - w
        # beside the error of any sum one rounding to a multiple of 2^-149
        assert np.linalg.norm(off) <= REL * np.linalg.norm(w) + 2.0 ** -150 * np.sqrt(w.size), name


def _poisoned(what, X, dY, rows, g):
    """rows: the kept rows; X, dY as wide as the layer's output and input"""
    inf, nan = float("inf"), float("nan")
    r = int(rows[5])
    if what == "one infinite row":
        X[r], dY[r] = inf, -inf
    elif what == "one NaN row":
        X[r], dY[r] = nan, nan
    elif what == "one infinite element":
        X[r, 3], dY[r, 7] = inf, inf
    elif what == "NaN":
        X.fill_(nan)
        dY.fill_(nan)
    elif what == "infinite":
        X.mul_(inf)
        dY.mul_(inf)
    else:                                            # finite, but beyond what the parts hold
        X.mul_(2.0 ** 114)
        dY.mul_(2.0 ** -20)


@pytest.mark.parametrize("what", ["one infinite row", "one NaN row", "one infinite element", "NaN", "infinite", "huge"])
@pytest.mark.parametrize("M,kept,C_in,C_out,out_in", [(3136, 1568, 768, 3072, False), (30000, 25001, 772, 260, True)])
def test_sums_that_are_made_again(M, kept, C_in, C_out, out_in, what):
    """Any share of sums that are not finite, at any depth: what the CUDA-core products give, for a bounded multiple of the finite call's time."""
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    X, dY = torch.randn(M, C_in, device="cuda", generator=g), torch.randn(M, C_out, device="cuda", generator=g)
    W = torch.randn(*((C_out, C_in) if out_in else (C_in, C_out)), device="cuda", generator=g) * C_in ** -0.5
    rows = torch.randperm(M, device="cuda", generator=g)[:kept].sort().values.int()
    flags = sbp.SBP_FLAG_W_OUT_IN if out_in else 0
    nb = sbp.sbp_linear_backward_workspace_bytes(sbp.SBP_F32, M, kept, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y, dW, db, dX = torch.empty(M, C_out, device="cuda"), torch.empty_like(W), torch.empty(C_out, device="cuda"), torch.empty_like(X)

    def call(extra=0):
        Xk = X[rows.long()]
        marks = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        marks[0].record()
        sbp.sbp_linear_forward(sbp.SBP_F32, X, W, None, M, C_in, C_out, Y, flags=flags | extra, status_word=status)
        marks[1].record()
        sbp.sbp_linear_backward(sbp.SBP_F32, Xk, dY, W, rows, None, M, kept, C_in, C_out, dW, db, dX, flags | extra, ws, nb, status)
        marks[2].record()
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        return np.array([marks[0].elapsed_time(marks[1]), marks[1].elapsed_time(marks[2])]), [t.clone() for t in (Y, dW, db, dX)]

    finite = np.min([call()[0] for _ in range(4)], axis=0)
    _poisoned(what, X, dY, rows, g)
    times, outs = zip(*[call() for _ in range(4)])
    # Measured: up to 9 times (all sums made again, none of them a NaN).  One thread a sum, without an early end, took 100 to 800 times.
    assert (np.min(times, axis=0) <= 25.0 * finite + 0.1).all(), (np.min(times, axis=0), finite)
    plain = call(sbp.SBP_FLAG_PLAIN_FMA)[1]
    for name, got, want in zip(("Y", "dW", "db", "dX"), outs[0], plain):
        assert torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isinf(), want.isinf()), name
        assert torch.equal(got[want.isinf()], want[want.isinf()]), name
        a, b = (torch.where(want.isfinite(), t, torch.zeros_like(t)).double() for t in (got, want))
        # two fp32 sums of the same terms: 2.5e-7 to 2e-6 (chains of FMAs) and below 3e-7 off
        assert float((a - b).norm()) <= 4e-6 * float(b.norm()), name


def test_more_items_than_a_launch_holds():
    """A worker notes sums to be made again for 1024 items; longer lists go in several launches.  Rows of either side of the cut, the first
    launch's last tile and the last, ragged one with a NaN in them."""
    M, C_in, C_out = 1024 * 74 * 256 + 300, 40, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(12)
    X, W = torch.randn(M, C_in, device="cuda", generator=g), torch.randn(C_in, C_out, device="cuda", generator=g)
    X[M - 400, 3] = X[M - 7, 5] = float("nan")
    Y = torch.full((M, C_out), 7.0, device="cuda")
    sbp.sbp_linear_forward(sbp.SBP_F32, X, W, None, M, C_in, C_out, Y)
    plain = torch.full((M, C_out), -7.0, device="cuda")
    sbp.sbp_linear_forward(sbp.SBP_F32, X, W, None, M, C_in, C_out, plain, flags=sbp.SBP_FLAG_PLAIN_FMA)
    torch.cuda.synchronize()
    bad = torch.zeros(M, dtype=torch.bool, device="cuda")
    bad[[M - 400, M - 7]] = True
    assert bool(Y[bad].isnan().all()) and not bool(Y[~bad].isnan().any())
    # sums of 40 terms of size 1 in two orders: below 40 * 2^-24 of the terms' sum of squares' root each
    Y[bad], plain[bad] = 0.0, 0.0
    assert float((Y - plain).abs().max()) <= 2 * 40 * 2.0 ** -24 * 40 ** 0.5
    assert float((Y - plain).norm() / plain.norm()) <= 3e-7


@pytest.mark.parametrize("kept,padding,C_in,C_out,out_in", [(1500, 0, 768, 3072, True), (1501, 77, 772, 3076, False)])
def test_bias_sums_of_one_piece_are_rounded_once(kept, padding, C_in, C_out, out_in):
    assert sbp.sbp_linear_backward_kernel_count(sbp.SBP_F32, 2 * kept, kept, C_in, C_out, 1, 1, 1, sbp.SBP_FLAG_W_OUT_IN if out_in else 0) == 1
    g = torch.Generator(device="cuda")
    g.manual_seed(13)
    M, valid = 2 * kept, kept - padding
    dY, X, W = (torch.randn(*s, device="cuda", generator=g) for s in ((M, C_out), (kept, C_in), (C_out, C_in) if out_in else (C_in, C_out)))
    rows = torch.randperm(M, device="cuda", generator=g)[:kept].sort().values.int()
    count = torch.tensor([valid], dtype=torch.int32, device="cuda") if padding else None
    _, db, _ = _backward(X, dY, W, rows, count, M, kept, C_in, C_out, sbp.SBP_FLAG_W_OUT_IN if out_in else 0, float("nan"))
    kept_dY = dY[rows[:valid].long()].double()
    want = kept_dY.sum(0)
    # half a unit in the last place, and what the sums of the rounding errors lose: each below 2^-24 of an error of 2^-24 of a partial sum
    bound = 2.0 ** -24 * want.abs() + valid * 2.0 ** -48 * kept_dY.abs().sum(0)
    assert bool(((db.double() - want).abs() <= bound).all())


@pytest.mark.parametrize("out_in", [False, True])
@pytest.mark.parametrize("wanted", ["dW", "dX", "dW db", "dX db", "dW dX", "db", "dW db dX"])
@pytest.mark.parametrize("M,kept,padding,C_in,C_out,on_cuda_cores", [
    (64, 32, 0, 2992, 352, {"dW", "dW db"}), (500, 254, 0, 1844, 72, {"dX", "dX db"}), (2000, 1081, 30, 164, 156, {"dW", "dW db", "dX", "dX db"}),
    (6000, 5000, 100, 260, 388, set()), (1500, 700, 0, 508, 516, set()),
])
def test_calls_for_some_of_the_outputs(M, kept, padding, C_in, C_out, on_cuda_cores, wanted, out_in):
    """dW or dX alone have a line of their own against the CUDA cores; every combination of outputs against the oracle, accumulated."""
    X, Wt, dY = synth.layer_inputs("f32", M, C_in, C_out, 95)
    keep = np.sort(np.random.default_rng(8).permutation(M)[:kept]).astype(np.int32)
    valid = keep[:kept - padding]
    rows, count = torch.from_numpy(keep).cuda(), torch.tensor([len(valid)], dtype=torch.int32, device="cuda")
    want = oracle.linear_backward(synth.to_f64(X[valid], "f32"), synth.to_f64(dY, "f32"), synth.to_f64(Wt, "f32"), valid)
    Xk, dY_d, W = dev(X[keep], "f32"), dev(dY, "f32"), dev(np.ascontiguousarray(Wt.T) if out_in else Wt, "f32")
    nb = sbp.sbp_linear_backward_workspace_bytes(sbp.SBP_F32, M, kept, C_in, C_out)
    results = []
    for extra in (0, sbp.SBP_FLAG_PLAIN_FMA):
        ws = torch.full((nb,), 0xff, dtype=torch.uint8, device="cuda")
        out = dict(dW=torch.full_like(W, 0.25), db=torch.full((C_out,), 0.25, device="cuda"), dX=torch.full((M, C_in), float("nan"), device="cuda"))
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        sbp.sbp_linear_backward(sbp.SBP_F32, Xk, dY_d, W, rows, count, M, kept, C_in, C_out, *(out[n] if n in wanted.split() else None for n in ("dW", "db", "dX")),
                                (sbp.SBP_FLAG_W_OUT_IN if out_in else 0) | sbp.SBP_FLAG_ACCUMULATE | extra, ws, nb, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        results.append(out)
    got, plain = results
    for name in wanted.split():
        g = host((got[name].t() if out_in and name == "dW" else got[name]).contiguous()).astype(np.float64)
        exact = want[name] + (0.0 if name == "dX" else 0.25)
        assert np.linalg.norm(g - exact) <= (1e-6 if wanted in on_cuda_cores else REL) * np.linalg.norm(exact), name
        same = torch.equal(got[name], plain[name])
        if name != "db":
            assert same == (wanted in on_cuda_cores), name
    for name in set(got) - set(wanted.split()):
        assert bool((got[name] == 0.25).all()) if name != "dX" else bool(got[name].isnan().all())
    if "dX" in wanted:
        assert not host(got["dX"])[np.setdiff1d(np.arange(M), valid)].view(np.uint8).any()
