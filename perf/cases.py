"""What is timed: calls of the public entry points as a user's program makes them, over the range the library is used in.

A case is one call (or, for the NVFP4 quantizer, the two calls its recipe takes) on tensors that are already where the
caller has them -- in device memory, or in pinned host memory for the host-buffer form -- with the workspace that such a
program keeps.  `op` names the entry point:

    mxfp4     forward_ws: the MXFP4 attention forward (options: UOS rule, PNQ row sum, Hadamard rotation, fp32 output)
    nvfp4     forward_nvfp4: the comparison format in the same fused forward
    bf16      forward_bf16: the unquantized high-precision forward
    host      forward_host: the MXFP4 forward on pinned host tensors, copies included
    quant     quantize_mxfp4_batched, canonical layout, block axis 1 (Q, K) or 0 (V)
    quant_nv  tensor_amax + quantize_nvfp4, canonical layout
"""
import math

import torch

import paper_2607_24377_b200 as mx

D = 128
SCALE = 1.0 / math.sqrt(D)


def _attn(name, op, B, H, Nq, Nkv, recipe, uos=True, pnq=True, hadamard=False, fp32=False):
    return {"name": name, "op": op, "B": B, "H": H, "Nq": Nq, "Nkv": Nkv, "recipe": recipe,
            "uos": uos, "pnq": pnq, "hadamard": hadamard, "fp32": fp32}


def _quant(name, op, batch, rows, cols, axis, recipe, uos=True):
    return {"name": name, "op": op, "batch": batch, "rows": rows, "cols": cols, "axis": axis, "recipe": recipe, "uos": uos}


def listed():
    return [
        # smallest forward: two heads of 1024 tokens, where launches and the latency of one KV tile after another count
        _attn("mxfp4_tiny", "mxfp4", 1, 2, 1024, 1024, "iid"),
        # ragged query and key counts, several batches, fp32 output: what a parity check or a small model's layer asks for
        _attn("mxfp4_ragged_fp32", "mxfp4", 2, 7, 1300, 777, "outlier", fp32=True),
        # all of Algorithm 2 (rotation of Q and K included) at the short end of the sequence sweep
        _attn("mxfp4_rotated_4k", "mxfp4", 1, 40, 4096, 4096, "outlier", hadamard=True),
        # the "MXFP4 (OCP)" baseline: floor rule, row sum from the unquantized exponentials
        _attn("mxfp4_ocp_8k", "mxfp4", 1, 24, 8192, 8192, "outlier", uos=False, pnq=False),
        # cross attention of a video model: long queries against a short text context
        _attn("mxfp4_cross", "mxfp4", 1, 40, 75600, 512, "wan"),
        # self attention of a 720p video model's layer, the size the library is meant for
        _attn("mxfp4_video_75600", "mxfp4", 1, 40, 75600, 75600, "wan"),
        # the comparison format with its own placement of the row sum
        _attn("nvfp4_16k", "nvfp4", 1, 40, 16384, 16384, "outlier", pnq=False),
        # the high-precision layer that a hybrid-precision policy keeps
        _attn("bf16_8k", "bf16", 1, 24, 8192, 8192, "outlier"),
        # tensors that live on the host: copies in, forward, copy out
        _attn("host_8k", "host", 1, 24, 8192, 8192, "outlier"),
        # one small tensor to quantize (1 Mi elements, blocks along the head dimension)
        _quant("quant_axis1_1m", "quant", 1, 8192, 128, 1, "iid"),
        # V of a long sequence, blocks along the tokens, transposed output (64 Mi elements)
        _quant("quant_axis0_64m", "quant", 16, 32768, 128, 0, "iid"),
        # the comparison format's quantizer: tensor maximum, then codes and scales (16 Mi elements)
        _quant("quant_nvfp4_axis1_16m", "quant_nv", 8, 16384, 128, 1, "outlier"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["mxfp4", "mxfp4", "mxfp4", "mxfp4", "mxfp4", "nvfp4", "bf16", "host", "quant", "quant", "quant_nv"])
    if op in ("quant", "quant_nv"):
        n = _log_int(rng, 1 << 19, 1 << 27)                       # elements
        batch = rng.choice([1, 1, 2, 5, 12, 24, 40])
        cols = rng.choice([128, 128, 128, 64, 256, 1024])
        rows = max(32, n // (batch * cols))
        return {"op": op, "batch": batch, "rows": rows, "cols": cols, "axis": rng.choice([0, 1]), "recipe": rng.choice(["iid", "outlier"]),
                "uos": rng.random() < 0.75}
    # 75600^2 pairs of 40 heads is the largest listed case; the slower forms get a smaller share of that
    most = {"mxfp4": 8.0e13, "nvfp4": 2.0e13, "bf16": 1.5e13, "host": 1.5e13}[op]
    H = rng.choice([1, 2, 3, 8, 12, 24, 24, 40, 40])
    B = rng.choice([1, 1, 1, 2, 4])
    Nq = _log_int(rng, 256, 76000 if op == "mxfp4" else 24000)
    kind = rng.random()
    Nkv = Nq if kind < 0.6 else (_log_int(rng, 77, 1024) if kind < 0.8 else _log_int(rng, 256, 32000))
    while 4.0 * B * H * Nq * Nkv * D > most:
        if B > 1:
            B //= 2
        elif H > 8:
            H //= 2
        else:
            Nq, Nkv = (int(0.8 * Nq), int(0.8 * Nkv))
    while B * H * (Nq + Nkv) > (2.5e6 if op == "host" else 6.5e6) and H > 1:     # the inputs stay below the largest listed case's
        H -= 1
    pnq = rng.random() < 0.7 if op != "nvfp4" else rng.random() < 0.4
    return {"op": op, "B": B, "H": H, "Nq": Nq, "Nkv": Nkv, "recipe": rng.choice(["iid", "outlier", "wan"]),
            "uos": pnq or rng.random() < 0.5, "pnq": pnq, "hadamard": op == "mxfp4" and rng.random() < 0.3,
            "fp32": op != "host" and rng.random() < 0.2}


# ---- inputs --------------------------------------------------------------------------------------
def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)


def _qkv(case, seed):
    """Q, K, V as the attention layers of the video models look: Gaussian; with a few large channels and a few large
    tokens ("outlier"); with a low-rank component that Q and K share and large channels ("wan")."""
    B, H, Nq, Nkv = case["B"], case["H"], case["Nq"], case["Nkv"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    q, k, v = _normal(g, B, H, Nq, D), _normal(g, B, H, Nkv, D), _normal(g, B, H, Nkv, D)
    if case["recipe"] == "outlier":
        ch = torch.randperm(D, generator=g, device="cuda")[:8]
        for x in (q, k):
            x[..., ch] *= 16.0
            n = x.shape[2]
            x[:, :, torch.randperm(n, generator=g, device="cuda")[:n // 100]] *= 8.0
    elif case["recipe"] == "wan":
        u = torch.linalg.qr(torch.randn(D, 4, generator=g, device="cuda"))[0].to(torch.bfloat16)
        ch = torch.randperm(D, generator=g, device="cuda")[:6]
        for x in (q, k):
            x += (2.0 * _normal(g, B, H, x.shape[2], 4)) @ u.T
            x[..., ch] *= 10.0
    return q, k, v


def _matrix(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = _normal(g, case["batch"], case["rows"], case["cols"])
    if case["recipe"] == "outlier":
        x[..., torch.randperm(case["cols"], generator=g, device="cuda")[:max(1, case["cols"] // 16)]] *= 16.0
    return x


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    op = case["op"]
    if op in ("quant", "quant_nv"):
        batch, rows, cols, axis = case["batch"], case["rows"], case["cols"], case["axis"]
        blk = 32 if op == "quant" else 16
        rp = -(-rows // 128) * 128
        shape = (lambda n: (batch, rows, cols // n)) if axis == 1 else (lambda n: (batch, cols, rp // n))
        s = {"x": _matrix(case, seed), "codes": _bytes(shape(2)), "scales": _bytes(shape(blk))}
        if op == "quant_nv":
            s["amax"] = torch.empty(batch, dtype=torch.float32, device="cuda")
            s["tensor_scale"] = torch.empty(batch, dtype=torch.float32, device="cuda")
        return {"case": case, **s}
    B, H, Nq, Nkv = case["B"], case["H"], case["Nq"], case["Nkv"]
    q, k, v = _qkv(case, seed)
    out = torch.float32 if case["fp32"] else torch.bfloat16
    flags = (mx.FLAG_OUT_FP32 if case["fp32"] else 0)
    if op == "bf16":
        ws = _bytes(mx.forward_bf16_workspace_bytes(B, H, Nq, Nkv, D))
    elif op == "nvfp4":
        flags |= mx.FLAG_PNQ if case["pnq"] else 0
        ws = _bytes(mx.forward_nvfp4_workspace_bytes(B, H, Nq, Nkv, D))
    else:
        flags |= (mx.FLAG_UOS if case["uos"] else 0) | (mx.FLAG_PNQ if case["pnq"] else 0) | (mx.FLAG_HADAMARD if case["hadamard"] else 0)
        ws = _bytes(mx.forward_host_arena_bytes(B, H, Nq, Nkv, D, flags) if op == "host" else mx.forward_workspace_bytes(B, H, Nq, Nkv, D))
    if op == "host":
        q, k, v = (x.to("cpu").pin_memory() for x in (q, k, v))
        o = torch.empty(q.shape, dtype=out).pin_memory()
    else:
        o = torch.empty(q.shape, dtype=out, device="cuda")
    return {"case": case, "q": q, "k": k, "v": v, "o": o, "ws": ws, "flags": flags}


# ---- one pass ------------------------------------------------------------------------------------
def run(s):
    c = s["case"]
    op = c["op"]
    if op == "quant":
        mx.quantize_mxfp4_batched(s["x"], s["codes"], s["scales"], c["batch"], c["rows"], c["cols"], c["axis"],
                                  mx.MODE_UOS if c["uos"] else mx.MODE_OCP, mx.LAYOUT_CANONICAL)
        return s["codes"], s["scales"]
    if op == "quant_nv":
        mx.tensor_amax(s["x"], s["amax"], c["batch"], c["rows"], c["cols"])
        mx.quantize_nvfp4(s["x"], s["codes"], s["scales"], s["amax"], s["tensor_scale"], c["batch"], c["rows"], c["cols"],
                          c["axis"], mx.LAYOUT_CANONICAL)
        return s["codes"], s["scales"], s["amax"], s["tensor_scale"]
    call = {"mxfp4": mx.forward_ws, "nvfp4": mx.forward_nvfp4, "bf16": mx.forward_bf16, "host": mx.forward_host}[op]
    call(s["q"], s["k"], s["v"], s["o"], c["B"], c["H"], c["Nq"], c["Nkv"], D, SCALE, s["flags"], s["ws"])
    return s["o"]


# ---- what a pass cannot do without, and how far two correct results may be apart ------------------
def work(case):
    if case["op"] in ("quant", "quant_nv"):
        n = case["batch"] * case["rows"] * case["cols"]
        out = case["batch"] * (-(-case["rows"] // 128) * 128 if case["axis"] == 0 else case["rows"]) * case["cols"]
        # the input once, codes and scales once
        return {"bytes": 2.0 * n + (0.5 + 1.0 / (32 if case["op"] == "quant" else 16)) * out, "flops": 0}
    B, H, Nq, Nkv = case["B"], case["H"], case["Nq"], case["Nkv"]
    return {"bytes": B * H * D * (2.0 * Nq + 4.0 * Nkv + (4.0 if case["fp32"] else 2.0) * Nq), "flops": 4.0 * B * H * Nq * Nkv * D}


def tolerance(case):
    if case["op"] in ("quant", "quant_nv"):
        return "exact"
    if case["op"] == "bf16":                    # probabilities and (by default) the output are bf16
        return {"rel": 5e-3, "max": 0.05}
    # fp32 sums; a probability next to a rounding boundary of its 4-bit grid may land on either side, which shows in the
    # few rows whose weight sits on a handful of keys; the bf16 output adds its own last place
    return {"rel": 2e-3 if case["fp32"] else 5e-3, "max": 0.5}
