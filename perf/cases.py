"""Performance cases: what a training program has the SBP library do in one step.

Four kinds of work, each through the public binding:

``block``      the layers of one block that share a keep set: draw the keep set, then per layer either the forward with
               its cache in one call (``sbp_linear_forward``) or only the cache (``sbp_forward_cache``, for programs whose
               own forward computes the layer), then the backward of every layer, last layer first.
``mlp``        the backward half of a d -> 4d -> d block whose gradient stays packed between the two layers.
``attention``  the backward of attention on token subsets, in the slices of a fused qkv projection.
``patch``      a stride = kernel convolution: patch cache, linear backward on patch rows, scatter.

Inputs follow the recipe of ``paper_2210_00129_b200.synth`` (X ~ N(0, 1), W ~ N(0, 0.02^2), dY ~ N(0, 1e-2^2); fp32
layers W ~ N(0, 1 / C_in), dY ~ N(0, 1)), drawn on the GPU from the seed.  All buffers, the workspace among them, belong
to the caller and are made once.
"""
from __future__ import annotations

import math

import torch

import paper_2210_00129_b200 as sbp

MODES = {"random": sbp.SBP_MASK_RANDOM, "grid": sbp.SBP_MASK_GRID, "frames": sbp.SBP_MASK_TEMPORAL,
         "frame_grid": sbp.SBP_MASK_TEMPORAL_GRID}
DTYPES = {"bf16": (sbp.SBP_BF16, torch.bfloat16, 2), "f32": (sbp.SBP_F32, torch.float32, 4)}


# ---- the listed cases ------------------------------------------------------------------------------------------------
def _block(name, dtype, mask, B, H, W, layers, ratio, forward, w_out_in, accumulate=False):
    return dict(name=name, kind="block", dtype=dtype, mask=mask, B=B, H=H, W=W, layers=layers, ratio=ratio,
                forward=forward, w_out_in=w_out_in, accumulate=accumulate)


def listed():
    return [
        # the smallest layer of the test-suite: six launches of a few microseconds each, bound by latency
        _block("fp32_smallest_layer", "f32", "random", 2, 16, 1, "32:64", 0.5, False, False),
        # one short clip per pass, whole frames kept, gradients accumulated over several passes: a small bf16 call
        _block("video_clip_accumulate", "bf16", "frames", 1, 8, 196, "768:768", 0.5, False, False, True),
        # a layer trained without mixed precision
        _block("fp32_mlp_layer_b16", "f32", "random", 16, 14, 14, "768:3072", 0.5, True, False),
        # the benchmark's workload: qkv, proj, fc1, fc2 of a ViT-B/16 block, keep ratio 0.5
        _block("vit_b16_block_b128", "bf16", "random", 128, 14, 14, "768:2304,768:768,768:3072,3072:768", 0.5, False, False),
        # the MLP of the same block where the library also runs the forward and weights are stored [C_out, C_in]
        _block("vit_b16_mlp_fwd_bwd_b64", "bf16", "random", 64, 14, 14, "768:3072,3072:768", 0.5, True, True),
        # point-wise pair of a ConvNeXt-B stage-1 block: few channels, many positions, grid masks (bound by memory)
        _block("convnext_b_s1_block_grid", "bf16", "grid", 64, 56, 56, "128:512,512:128", 0.5, False, False),
        # stage 4: many channels on ragged 7 x 7 maps (24 or 25 kept positions each, counted on the device)
        _block("convnext_b_s4_fwd_bwd_ragged", "bf16", "grid", 64, 7, 7, "1024:4096,4096:1024", 0.5, True, True),
        # detection resolution: two images of 200 x 334 positions
        _block("detection_block_200x334", "bf16", "random", 2, 200, 334, "128:512,512:128", 0.5, False, False),
        # a whole MLP backward packed from end to end at the largest batch
        dict(name="vit_b16_mlp_packed_b256", kind="mlp", dtype="bf16", mask="random", B=256, H=14, W=14, C=768, hidden=3072,
             ratio=0.5),
        # attention inside a block that drops the same tokens everywhere (queries, keys and values)
        dict(name="attention_drop_qkv_b128", kind="attention", B=128, H=14, W=14, heads=12, ratio=0.5, keys="kept",
             kept_rows_only=False),
        # attention that keeps all keys and values and drops queries only
        dict(name="attention_drop_query_b64", kind="attention", B=64, H=14, W=14, heads=12, ratio=0.5, keys="all",
             kept_rows_only=False),
        # ConvNeXt-B down-sampling between stages 1 and 2: 2 x 2 / stride 2
        dict(name="convnext_b_downsample_b64", kind="patch", dtype="bf16", mask="random", B=64, H=56, W=56, C=128,
             C_out=256, k=2, ratio=0.5),
    ]


# ---- more cases of the same ranges -----------------------------------------------------------------------------------
def _log_int(rng, lo, hi, step=1):
    """An integer of [lo, hi], a multiple of `step`, spread evenly over its logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def _width(rng, lo, hi):
    """A channel count: usually a multiple of 64, otherwise only of 8."""
    return _log_int(rng, lo, hi, 64 if lo % 64 == 0 and rng.random() < 0.7 else 8)


def _ratio(rng, mask):
    return rng.choice([0.25, 0.5, 0.75, 1.0]) if mask.endswith("grid") or rng.random() < 0.5 else round(rng.uniform(0.1, 0.9), 2)


def _map(rng, most):
    """Height and width of a feature map of at most `most` positions, odd sizes among them."""
    H = _log_int(rng, 5, int(math.sqrt(most)))
    return H, max(4, min(most // H, _log_int(rng, max(4, H // 2), 2 * H)))


def _draw_block(rng):
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    mask = rng.choice(["random", "random", "random", "grid", "grid", "frames", "frame_grid"])
    if mask.startswith("frame"):
        H, W = _log_int(rng, 4, 32), rng.choice([49, 100, 196, 256])
        B = _log_int(rng, 1, 8)
    else:
        H, W = _map(rng, 80000 if rng.random() < 0.15 else 4096)
        B = _log_int(rng, 1, 256)
    a, b = (_width(rng, 32, 1024), _width(rng, 32, 3072)) if dtype == "f32" else (_width(rng, 64, 4096), _width(rng, 64, 4096))
    pair = rng.random() < 0.5
    return dict(kind="block", dtype=dtype, mask=mask, B=B, H=H, W=W, layers=f"{a}:{b},{b}:{a}" if pair else f"{a}:{b}",
                ratio=_ratio(rng, mask), forward=rng.random() < 0.5, w_out_in=rng.random() < 0.4, accumulate=rng.random() < 0.2)


def _draw_mlp(rng):
    mask = rng.choice(["random", "grid"])
    H, W = _map(rng, 4096)
    C = _width(rng, 64, 1280)
    return dict(kind="mlp", dtype="bf16", mask=mask, B=_log_int(rng, 2, 256), H=H, W=W, C=C, hidden=4 * C, ratio=_ratio(rng, mask))


def _draw_attention(rng):
    H, W = _map(rng, 256)
    return dict(kind="attention", B=_log_int(rng, 1, 192), H=H, W=W, heads=_log_int(rng, 2, 20), ratio=_ratio(rng, "random"),
                keys=rng.choice(["kept", "kept", "all"]), kept_rows_only=rng.random() < 0.3)


def _draw_patch(rng):
    k = rng.choice([2, 2, 4])
    H, W = _map(rng, 4096)
    mask = rng.choice(["random", "grid"])
    return dict(kind="patch", dtype="bf16", mask=mask, B=_log_int(rng, 2, 128), H=k * max(4, H // k), W=k * max(4, W // k),
                C=_width(rng, 32, 512) if k == 2 else _log_int(rng, 8, 64, 8), C_out=_width(rng, 64, 1024), k=k,
                ratio=_ratio(rng, mask))


def _cost(case):
    """Rough seconds of one pass, to keep drawn cases below the largest listed one (fp32 layers and layers below 128
    channels at the rate of the CUDA cores)."""
    w = work(case)
    widths = [v for pair in _layers(case) for v in pair] if case["kind"] == "block" else [case.get("C", 128)]
    slow = case.get("dtype") == "f32" or (case["kind"] != "patch" and min(widths) < 128)
    return max(w["flops"] / (20e12 if slow else 700e12), w["bytes"] / 4e12)


def draw(rng):
    limit = max(_cost(c) for c in listed())
    while True:
        case = rng.choice([_draw_block, _draw_block, _draw_block, _draw_mlp, _draw_attention, _draw_patch])(rng)
        if _cost(case) <= limit:
            return case


# ---- sizes -----------------------------------------------------------------------------------------------------------
def _layers(case):
    return [tuple(int(v) for v in part.split(":")) for part in case["layers"].split(",")]


def _grid_of(case):
    """Positions the keep set chooses among: of the output for a strided convolution."""
    k = case.get("k", 1)
    return case["H"] // k, case["W"] // k


def _kept(case):
    """(rows of all samples, most rows kept)"""
    H, W = _grid_of(case)
    return case["B"] * H * W, case["B"] * sbp.sbp_keep_count(MODES[case.get("mask", "random")], H, W, case["ratio"])


def work(case):
    M, kept = _kept(case)
    es = 4 if case.get("dtype") == "f32" else 2
    kind, by, flops = case["kind"], 4.0 * kept, 0.0

    def backward(ci, co, dx_rows, accumulate=False):
        return es * (kept * (ci + co) + ci * co + dx_rows * ci) + (8 if accumulate else 4) * (ci + 1) * co, 4.0 * kept * ci * co

    if kind == "block":
        for ci, co in _layers(case):
            b, f = backward(ci, co, M, case["accumulate"])
            if case["forward"]:
                b += es * (M * ci + ci * co + M * co + kept * ci) + 4 * co
                f += 2.0 * M * ci * co
            else:
                b += es * 2 * kept * ci
            by, flops = by + b, flops + f
    elif kind == "mlp":
        C, h = case["C"], case["hidden"]
        b2, f2 = backward(h, C, kept)
        b1, f1 = backward(C, h, M)
        by += es * 2 * kept * (C + 2 * h) + b2 + es * 3 * kept * h + b1
        flops += f1 + f2
    elif kind == "attention":
        width, n, q = 64 * case["heads"], case["H"] * case["W"], kept // case["B"]
        keys = n if case["keys"] == "all" else q
        q_out, k_out = (q, keys) if case["kept_rows_only"] else (n, n)
        by += 2.0 * case["B"] * width * (2 * q + 2 * keys + q_out + 2 * k_out)
        flops += 10.0 * case["B"] * width * q * keys
    else:
        ci, co = case["k"] ** 2 * case["C"], case["C_out"]
        b, f = backward(ci, co, kept)
        by += es * (2 * kept * ci + kept * ci + case["B"] * case["H"] * case["W"] * case["C"]) + b
        flops += f
    return {"bytes": by, "flops": flops}


# ---- a program's state and one pass over it --------------------------------------------------------------------------
class _Gpu:
    """Tensors on the GPU, drawn from one seeded stream."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, dtype, *shape, sigma=1.0):
        t = torch.randn(*shape, device="cuda", dtype=torch.float32, generator=self.gen)
        return t.mul_(sigma).to(DTYPES[dtype][1])

    @staticmethod
    def zeros(tdt, *shape):
        return torch.zeros(*shape, device="cuda", dtype=tdt)


def _linear(gpu, case, ci, co, M, kept):
    """Weights, output gradients and workspace of one layer."""
    code, tdt, _ = DTYPES[case["dtype"]]
    fp32 = case["dtype"] == "f32"
    shape = (co, ci) if case.get("w_out_in") else (ci, co)
    nbytes = sbp.sbp_linear_backward_workspace_bytes(code, M, kept, ci, co)
    return dict(ci=ci, co=co, W=gpu.normal(case["dtype"], *shape, sigma=ci ** -0.5 if fp32 else 0.02),
                dW=gpu.zeros(torch.float32, *shape), db=gpu.zeros(torch.float32, co),
                ws=torch.empty(nbytes, dtype=torch.uint8, device="cuda"), nbytes=nbytes)


def prepare(case, seed):
    gpu = _Gpu(seed)
    M, kept = _kept(case)
    dtype = case.get("dtype", "bf16")
    code, tdt, _ = DTYPES[dtype]
    sigma_dy = 1.0 if dtype == "f32" else 1e-2
    mask = case.get("mask", "random")
    s = dict(case=case, kind=case["kind"], code=code, mode=MODES[mask], M=M, kept=kept, seed=seed, step=seed % 100000,
             grid=_grid_of(case), rows=gpu.zeros(torch.int32, kept), offs=gpu.zeros(torch.int32, case["B"] + 1),
             status=gpu.zeros(torch.int32, 1))
    # grid masks keep a number of rows that only the device knows
    s["count"] = s["offs"][case["B"]:] if mask.endswith("grid") else None
    if case["kind"] == "block":
        s["flags"] = (sbp.SBP_FLAG_W_OUT_IN if case["w_out_in"] else 0) | (sbp.SBP_FLAG_ACCUMULATE if case["accumulate"] else 0)
        s["layers"] = []
        for ci, co in _layers(case):
            L = _linear(gpu, case, ci, co, M, kept)
            L.update(X=gpu.normal(dtype, M, ci), dY=gpu.normal(dtype, M, co, sigma=sigma_dy), Xk=gpu.zeros(tdt, kept, ci),
                     dX=gpu.zeros(tdt, M, ci))
            if case["forward"]:
                L.update(bias=gpu.normal("f32", co, sigma=0.1), Y=gpu.zeros(tdt, M, co))
            s["layers"].append(L)
    elif case["kind"] == "mlp":
        C, h = case["C"], case["hidden"]
        fc1, fc2 = _linear(gpu, case, C, h, M, kept), _linear(gpu, case, h, C, M, kept)
        Z = gpu.normal(dtype, M, h)                      # what the program's own forward left: fc1's output, its GELU
        fc1.update(X=gpu.normal(dtype, M, C), Xk=gpu.zeros(tdt, kept, C), dX=gpu.zeros(tdt, M, C))
        fc2.update(X=torch.nn.functional.gelu(Z), Xk=gpu.zeros(tdt, kept, h), dX=gpu.zeros(tdt, kept, h))
        s.update(fc1=fc1, fc2=fc2, Z=Z, Zk=gpu.zeros(tdt, kept, h), dZ=gpu.zeros(tdt, kept, h), dY=gpu.normal(dtype, M, C, sigma=sigma_dy))
    elif case["kind"] == "attention":
        C = 64 * case["heads"]
        qkv, grad = gpu.normal(dtype, M, 3 * C), gpu.zeros(tdt, M, 3 * C)
        s.update(C=C, qkv=[qkv[:, i * C:] for i in range(3)], dA=gpu.normal(dtype, M, C, sigma=1e-2), grad=grad,
                 dqkv=[grad[:, i * C:] for i in range(3)], most=kept // case["B"],
                 flags=(sbp.SBP_FLAG_ATTN_ALL_KEYS if case["keys"] == "all" else 0) |
                       (sbp.SBP_FLAG_ATTN_KEPT_ROWS_ONLY if case["kept_rows_only"] else 0))
    else:
        B, H, W, C, k = (case[n] for n in ("B", "H", "W", "C", "k"))
        ci, co = k * k * C, case["C_out"]
        L = _linear(gpu, case, ci, co, M, kept)
        nbytes = sbp.sbp_patch_scatter_workspace_bytes(B, H, W, k, k)
        L.update(X=gpu.normal(dtype, B, H, W, C), dY=gpu.normal(dtype, M, co, sigma=sigma_dy), Xk=gpu.zeros(tdt, kept, ci),
                 dXp=gpu.zeros(tdt, kept, ci), dX=gpu.zeros(tdt, B, H, W, C),
                 ws2=torch.empty(nbytes, dtype=torch.uint8, device="cuda"), nbytes2=nbytes)
        s["layer"] = L
    return s


def _draw_keep_set(s):
    H, W = s["grid"]
    sbp.sbp_sample_keep(s["mode"], s["case"]["B"], H, W, s["case"]["ratio"], s["seed"], s["step"], 0, 0, s["rows"], s["offs"])


def _run_block(s):
    code, M, kept, rows, count, status = s["code"], s["M"], s["kept"], s["rows"], s["count"], s["status"]
    forward = s["case"]["forward"]
    _draw_keep_set(s)
    for L in s["layers"]:
        if forward:
            sbp.sbp_linear_forward(code, L["X"], L["W"], L["bias"], M, L["ci"], L["co"], L["Y"], rows, count, kept, L["Xk"],
                                   s["flags"] & sbp.SBP_FLAG_W_OUT_IN, status)
        else:
            sbp.sbp_forward_cache(code, L["X"], M, L["ci"], rows, count, kept, L["Xk"])
    for L in reversed(s["layers"]):
        sbp.sbp_linear_backward(code, L["Xk"], L["dY"], L["W"], rows, count, M, kept, L["ci"], L["co"], L["dW"], L["db"], L["dX"],
                                s["flags"], L["ws"], L["nbytes"], status)
    names = ("Y", "Xk", "dW", "db", "dX") if forward else ("Xk", "dW", "db", "dX")
    return [rows, s["offs"], [[L[n] for n in names] for L in s["layers"]]]


def _run_mlp(s):
    code, M, kept, rows, count, status, fc1, fc2 = (s[n] for n in ("code", "M", "kept", "rows", "count", "status", "fc1", "fc2"))
    _draw_keep_set(s)
    sbp.sbp_forward_cache(code, fc1["X"], M, fc1["ci"], rows, count, kept, fc1["Xk"])
    sbp.sbp_forward_cache(code, s["Z"], M, fc1["co"], rows, count, kept, s["Zk"])
    sbp.sbp_forward_cache(code, fc2["X"], M, fc2["ci"], rows, count, kept, fc2["Xk"])
    sbp.sbp_linear_backward(code, fc2["Xk"], s["dY"], fc2["W"], rows, count, M, kept, fc2["ci"], fc2["co"], fc2["dW"], fc2["db"],
                            fc2["dX"], sbp.SBP_FLAG_DX_COMPACT, fc2["ws"], fc2["nbytes"], status)
    sbp.sbp_act_backward(code, sbp.SBP_ACT_GELU, s["Zk"], fc2["dX"], count, kept, fc1["co"], s["dZ"], status)
    sbp.sbp_linear_backward(code, fc1["Xk"], s["dZ"], fc1["W"], rows, count, M, kept, fc1["ci"], fc1["co"], fc1["dW"], fc1["db"],
                            fc1["dX"], sbp.SBP_FLAG_DY_COMPACT, fc1["ws"], fc1["nbytes"], status)
    return [rows, [[L[n] for n in ("Xk", "dW", "db", "dX")] for L in (fc1, fc2)], s["Zk"], s["dZ"]]


def _run_attention(s):
    case, (q, k, v), (dq, dk, dv), C = s["case"], s["qkv"], s["dqkv"], s["C"]
    _draw_keep_set(s)
    sbp.sbp_attention_backward(s["code"], q, k, v, 3 * C, s["dA"], C, s["rows"], s["offs"], None, None, case["B"],
                               case["H"] * case["W"], case["heads"], 64, s["most"], dq, dk, dv, 3 * C, s["flags"], s["status"])
    return [s["rows"], s["grad"]]


def _run_patch(s):
    case, L, code, kept, rows, count = s["case"], s["layer"], s["code"], s["kept"], s["rows"], s["count"]
    B, H, W, C, k = (case[n] for n in ("B", "H", "W", "C", "k"))
    _draw_keep_set(s)
    sbp.sbp_patch_cache(code, L["X"], B, H, W, C, k, k, rows, count, kept, L["Xk"])
    sbp.sbp_linear_backward(code, L["Xk"], L["dY"], L["W"], rows, count, s["M"], kept, L["ci"], L["co"], L["dW"], L["db"], L["dXp"],
                            sbp.SBP_FLAG_DX_COMPACT, L["ws"], L["nbytes"], s["status"])
    sbp.sbp_patch_scatter(code, L["dXp"], B, H, W, C, k, k, rows, count, kept, L["dX"], L["ws2"], L["nbytes2"], s["status"])
    return [rows, [L[n] for n in ("Xk", "dW", "db", "dXp", "dX")]]


_RUN = {"block": _run_block, "mlp": _run_mlp, "attention": _run_attention, "patch": _run_patch}


def run(state):
    return _RUN[state["kind"]](state)


def tolerance(case):
    # Four times what the pass shows against the same arithmetic in 64 bits, as the largest of all outputs of the listed
    # cases and a dozen drawn ones (relative 2-norm / largest element): fp32 layers 1.0e-6 / 9.5e-6; bf16 layers and
    # convolutions 1.7e-3 / 3.9e-3 (one rounding of Y or dX to bf16); the packed MLP 2.9e-3 / 2.6e-2 and attention
    # 2.4e-3 / 3.3e-2 (bf16 intermediates).
    if case.get("dtype") == "f32":
        return {"rel": 5e-6, "max": 5e-5}
    if case["kind"] == "mlp":
        return {"rel": 1.2e-2, "max": 0.1}
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 0.13}
    return {"rel": 7e-3, "max": 1.6e-2}
