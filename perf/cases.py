"""Workloads of the quantized linear path, as a program that serves the transformer blocks runs them.

A case names a path through the public entry points, the linears it runs (K x N, in order) and the number of token rows:

    path      c8        4-bit codes one per byte, exact quantize kernel, per-token scales (the default way to run a layer)
              packed    4-bit codes two per byte for activations and weights
              expand    activations one code per byte; the handle keeps packed weights, expanded by the quantize launch
              w8a8      8-bit codes
              tc        as c8 with the tensor-core Hadamard mode of the quantize kernel
              group128  as c8 with one activation scale per 128 rotated channels
              static    as c8 with one given step size for the whole activation tensor
              fused     as c8 with the producers of a block fused in front: LayerNorm before qkv and fc1, GELU before fc2
              load      offline: smoothing factors from a calibration batch, weights folded, quantized and stored
    linears   "KxN+KxN+...": 1024x3072 = qkv, 1024x1024 = proj, 1024x4096 = fc1, 4096x1024 = fc2
    tokens    rows M (a frame is 1374 tokens, five of them special; load: rows of the calibration batch)
    pad       extra elements between activation rows (X is a column slice of a wider tensor when > 0)

Every case returns the outputs of all its calls: codes, scales and bf16 results (load: factors, codes, scales, multipliers).
"""
import math

import torch

import paper_2509_21302_b200 as q

FRAME = 1374
SPECIAL = 5
BLOCK = "1024x3072+1024x1024+1024x4096+4096x1024"
MLP = "1024x4096+4096x1024"
PATHS = ("c8", "packed", "expand", "w8a8", "tc", "group128", "static", "fused", "load")
MAX_FLOPS = 2.0 * 100 * FRAME * 2 * 1024 * 4096     # the largest listed case: both MLP linears over a 100-frame scene


def listed():
    return [
        # the five special tokens of one frame through one projection: the smallest call, two launches
        dict(name="special_tokens_proj", path="c8", linears="1024x1024", tokens=SPECIAL, pad=0),
        # one frame through one projection: latency of a single layer
        dict(name="frame_proj", path="c8", linears="1024x1024", tokens=FRAME, pad=0),
        # one frame and a ragged rest through a whole block, static step size, input sliced out of a wider tensor
        dict(name="block_ragged_static", path="static", linears=BLOCK, tokens=FRAME + 77, pad=64),
        # two frames less a few tokens through a block in the packed storage format
        dict(name="block_2f_packed", path="packed", linears=BLOCK, tokens=2 * FRAME - 17, pad=0),
        # three frames, weights kept at half a byte each and expanded on the way
        dict(name="block_3f_expand", path="expand", linears=BLOCK, tokens=3 * FRAME, pad=0),
        # the eight-frame block of the benchmark, in its default format
        dict(name="block_8f", path="c8", linears=BLOCK, tokens=8 * FRAME, pad=0),
        # the same block with the normalization and the activation fused in front of the quantize kernels
        dict(name="block_8f_fused", path="fused", linears=BLOCK, tokens=8 * FRAME, pad=0),
        # the paper's 8-bit setting
        dict(name="block_8f_w8a8", path="w8a8", linears=BLOCK, tokens=8 * FRAME, pad=0),
        # 32 frames (the multi-view setting of the 48-block stack) with the tensor-core quantize mode
        dict(name="block_32f_tc", path="tc", linears=BLOCK, tokens=32 * FRAME, pad=0),
        # group-wise activation scales through the MLP at 32 frames
        dict(name="mlp_32f_group128", path="group128", linears=MLP, tokens=32 * FRAME, pad=0),
        # the MLP over a 100-frame scene: the largest call
        dict(name="mlp_100f", path="c8", linears=MLP, tokens=100 * FRAME, pad=0),
        # preparing one block's four linears from bf16 weights and one frame of calibration activations
        dict(name="load_block", path="load", linears=BLOCK, tokens=FRAME, pad=0),
    ]


def draw(rng):
    path = rng.choice(PATHS)
    kinds = ["1024x3072", "1024x1024", "1024x4096", "4096x1024"]
    r = rng.random()
    if r < 0.35:
        linears = BLOCK
    elif r < 0.5:
        linears = MLP
    elif r < 0.8:
        linears = rng.choice(kinds)
    else:                                            # any N is a multiple of 128
        linears = "%dx%d" % (rng.choice((1024, 4096)), 128 * rng.randint(1, 32))
    per_token = sum(2.0 * k * n for k, n in _shapes(linears))
    hi = min(100 * FRAME, int(MAX_FLOPS / per_token))
    if path == "load":
        tokens = rng.randint(64, 2 * FRAME)
    else:
        tokens = int(round(math.exp(rng.uniform(0.0, math.log(hi)))))
        if rng.random() < 0.3 and tokens >= FRAME:   # whole frames are as common as ragged batches
            tokens -= tokens % FRAME
    pad = rng.choice((0, 0, 0, 8, 64, 1024)) if path != "load" else 0
    return dict(path=path, linears=linears, tokens=max(1, min(hi, tokens)), pad=pad)


def _shapes(linears):
    return [tuple(int(v) for v in s.split("x")) for s in linears.split("+")]


def _activations(g, M, K, pad, kind):
    """Token rows with outlier channels (x50) and large special tokens (x100, the first five of every frame); `kind`: the
    producer of the tensor -- "normal", "gelu" (after the activation function) or "pre" (in front of it)."""
    x = torch.empty((M, K + pad), dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 26) // (K + pad))
    outlier = torch.randperm(K, generator=g, device="cuda")[:8]
    for m0 in range(0, M, rows):
        m1 = min(M, m0 + rows)
        v = torch.empty((m1 - m0, K + pad), dtype=torch.float32, device="cuda").normal_(generator=g)
        if kind == "pre":
            v *= 1.5
        else:
            if kind == "gelu":
                v = torch.nn.functional.gelu(v * 1.5)
            v[:, outlier] *= 50.0
            special = torch.arange(m0, m1, device="cuda") % FRAME < SPECIAL
            v *= torch.where(special, 100.0, 1.0)[:, None]
        x[m0:m1] = v
    return x[:, :K]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    path, M, pad = case["path"], case["tokens"], case["pad"]
    layers = []
    for K, N in _shapes(case["linears"]):
        W = (torch.empty((N, K), dtype=torch.float32, device="cuda").normal_(generator=g) * 0.02).to(torch.bfloat16)
        b = (torch.empty((N,), dtype=torch.float32, device="cuda").normal_(generator=g) * 0.01).to(torch.bfloat16)
        after_mlp = K == 4096
        if path == "load":
            layers.append(dict(W=W, b=b, calib=_activations(g, M, K, 0, "gelu" if after_mlp else "normal")))
            continue
        c = q.calibrate_smooth(_activations(g, 256, K, 0, "gelu" if after_mlp else "normal").contiguous(), W)
        if path in ("packed", "expand"):
            h = q.prepare_weights(W, b, c, None)
        elif path == "w8a8":
            h = q.prepare_weights(W, b, c, None, bits=8)
        else:
            h = q.prepare_weights(W, b, c, None, c8="only")
        kind = ("pre" if path == "fused" else "gelu") if after_mlp else "normal"
        L = dict(h=h, K=K, N=N, x=_activations(g, M, K, pad, kind),
                 y=torch.empty((M, N), dtype=torch.bfloat16, device="cuda"),
                 a=torch.empty((M, K // 128) if path == "group128" else (M,), dtype=torch.float32, device="cuda"),
                 xq=torch.empty((M, K // 2), dtype=torch.uint8, device="cuda") if path == "packed" else
                 torch.empty((M, K), dtype=torch.int8, device="cuda"))
        if path == "static":          # one step size, from a calibration batch
            _, a = q.rotate_smooth_quantize_c8(h, _activations(g, 256, K, 0, kind))
            L["delta"] = a.max().reshape(1).clone()
        if path == "fused" and not after_mlp and N > 1024:      # the block's two normalized linears
            L["gamma"] = torch.empty((K,), dtype=torch.float32, device="cuda").normal_(1.0, 0.1, generator=g)
            L["beta"] = torch.empty((K,), dtype=torch.float32, device="cuda").normal_(0.0, 0.1, generator=g)
        layers.append(L)
    state = dict(path=path, layers=layers)
    if path == "expand":              # one scratch serves every layer of the stream
        state["scratch"] = torch.empty((max(L["N"] * L["K"] for L in layers),), dtype=torch.int8, device="cuda")
    return state


def run(state):
    path, out = state["path"], []
    for L in state["layers"]:
        if path == "load":
            c = q.calibrate_smooth(L["calib"], L["W"])
            h = q.prepare_weights(L["W"], L["b"], c, None, c8="only")
            codes, v = h.view_c8(), h.view()
            out += [c, codes, v["w_scale"], v["amul"]]
            h.free()
            continue
        h, x, xq, a, y = L["h"], L["x"], L["xq"], L["a"], L["y"]
        if path == "packed":
            q.rotate_smooth_quantize(h, x, 0, xq, a)
            q.w4a4_linear(h, xq, a, 0, y)
        elif path == "expand":
            q.rotate_smooth_quantize_c8_expand(h, x, state["scratch"], xq, a)
            q.w4a4_linear_c8_expanded(h, xq, a, state["scratch"], y)
        elif path == "group128":
            q.rotate_smooth_quantize_c8_grouped(h, x, xq, a)
            q.w4a4_linear_c8_grouped(h, xq, a, y)
        else:
            if path == "tc":
                q.rotate_smooth_quantize_tc(h, x, True, xq, a)
            elif path == "static":
                q.rotate_smooth_quantize_static_c8(h, x, L["delta"], xq, a)
            elif "gamma" in L:
                q.layernorm_rotate_smooth_quantize_c8(h, x, L["gamma"], L["beta"], 1e-5, xq, a)
            elif path == "fused" and L["K"] == 4096:
                q.gelu_rotate_smooth_quantize_c8(h, x, xq, a)
            else:
                q.rotate_smooth_quantize_c8(h, x, xq, a)
            q.w4a4_linear_c8(h, xq, a, y)
        out += [xq, a, y]
    return out


def work(case):
    """Each input read once, each returned output written once; integer multiply-adds of the products (load: the additions of the
    rotations, which is all there is)."""
    path, M = case["path"], case["tokens"]
    nbytes = flops = 0.0
    for K, N in _shapes(case["linears"]):
        if path == "load":
            # weights and calibration rows in; codes, scales, multipliers and factors out
            nbytes += 2.0 * N * K + 2.0 * M * K + N * K + 4 * N + 8 * K + 4 * N
            flops += (2.0 * N + M) * K * math.log2(K)
            continue
        code = 0.5 if path == "packed" else 1.0
        wcode = 0.5 if path in ("packed", "expand") else 1.0
        groups = K // 128 if path == "group128" else 1
        nbytes += M * (2.0 * K + K * code + 4 * groups + 2.0 * N) + N * K * wcode + 6.0 * N + 4.0 * K
        flops += 2.0 * M * N * K
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """Codes, scales and results are fixed bit for bit by the stated order of the operations, except where the interface
    leaves the arithmetic open.  Measured at 64, 1374 and 10 992 rows, about four times the largest seen:
    tc      against the exact kernel: results 4.5e-5 (largest single value 1.2e-2 of the rms), scales 8e-8, 9e-8 of the codes
    fused   GELU against its value in 64 bits, rounded to bf16: results 8e-3 (0.25), scales 1.2e-6, 8e-6 of the codes; LayerNorm is exact
    load    the smoothing factors off by 2e-7: scales 2e-7 (9e-7), 1e-6 of the codes"""
    if case["path"] == "tc":
        return dict(rel=2e-4, max=0.05, differ=1e-6)
    if case["path"] == "fused" and "4096x" in case["linears"]:
        return dict(rel=2e-2, max=0.9, differ=4e-5)
    if case["path"] == "load":
        return dict(rel=1e-6, max=4e-6, differ=4e-6)
    return "exact"
