"""Performance cases of the CLEAR attention library: the calls a model makes, through the Python binding.

A diffusion transformer calls this library once per attention layer and step: it prepares Q and K
(``clear_qk_norm_rope``), runs the attention forward (``clear_attn_fwd``), and when it is distilled, the backward
pass (``clear_attn_bwd_bf16_tc``).  The fp32 entry points serve evaluation at full precision and gradient checks of
small problems; ``Plan.forward_host`` serves callers whose tensors live in pinned host memory.

A case names an operation, a data type and a shape: B x H heads of ``head_dim`` channels over ``n_text`` text tokens
and a ``grid_h`` x ``grid_w`` latent grid (image resolution / 16), with window radius ``radius``.
"""
from __future__ import annotations

import math

import torch

from paper_2412_16112_b200 import binding as clear

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, op, dtype, B, H, grid_h, grid_w, n_text, head_dim, radius):
    return {"name": name, "op": op, "dtype": dtype, "B": B, "H": H, "grid_h": grid_h, "grid_w": grid_w,
            "n_text": n_text, "head_dim": head_dim, "radius": float(radius)}


def listed():
    return [
        # the tiny fp32 configuration of the repository: the smallest call, bound by launch and latency
        _case("fwd_f32_tiny", "forward", "f32", 1, 2, 16, 16, 16, 64, 4),
        # a 1024px layer evaluated in fp32 (reference outputs for a bf16 model)
        _case("fwd_f32_1024px_r8", "forward", "f32", 1, 24, 64, 64, 512, 128, 8),
        # inference at the paper's training resolution: the ordinary call
        _case("fwd_1024px_r8", "forward", "bf16", 1, 24, 64, 64, 512, 128, 8),
        # a landscape picture whose grid divides into no tile, conditional and unconditional half in one batch,
        # 64-channel heads, a text length that fills no tile, a fractional radius
        _case("fwd_67x120_ragged_d64", "forward", "bf16", 2, 12, 67, 120, 300, 64, 12.5),
        # high-resolution inference, with the radii the paper lists for them
        _case("fwd_2048px_r16", "forward", "bf16", 1, 24, 128, 128, 512, 128, 16),
        _case("fwd_4096px_r32", "forward", "bf16", 1, 24, 256, 256, 512, 128, 32),
        # the headline workload, the largest call
        _case("fwd_8k_r16", "forward", "bf16", 1, 24, 512, 512, 512, 128, 16),
        # what a layer does between its projections: normalise and rotate Q and K, then attend
        _case("layer_1024px_r16", "layer", "bf16", 1, 24, 64, 64, 512, 128, 16),
        # distillation: backward pass at the training resolution, and of a high-resolution layer
        _case("bwd_1024px_r8", "backward", "bf16", 1, 24, 64, 64, 512, 128, 8),
        _case("bwd_2048px_r16", "backward", "bf16", 1, 24, 128, 128, 512, 128, 16),
        # fp32 gradients of a small problem (gradient checks, small models)
        _case("bwd_f32_24x40_r8", "backward", "f32", 1, 24, 24, 40, 130, 64, 8),
        # a caller with its tensors in pinned host memory: copies in, kernels, copy out
        _case("host_1024px_r8", "forward_host", "bf16", 1, 24, 64, 64, 512, 128, 8),
    ]


def _sum_mask(c):
    """Allowed (query, key) pairs of one head: text rows and columns in full, image pairs closer than the radius."""
    gh, gw, T = c["grid_h"], c["grid_w"], c["n_text"]
    n, limit = gh * gw, math.ceil(c["radius"] ** 2)  # dx^2 + dy^2 < limit, whole numbers
    pairs = 0
    for dy in range(gh):
        left = limit - 1 - dy * dy
        if left < 0:
            break
        m = min(math.isqrt(left), gw - 1)
        pairs += (1 if dy == 0 else 2) * (gh - dy) * (gw * (2 * m + 1) - m * (m + 1))
    return T * (T + n) + n * T + pairs


def _flops(c):
    products = 10 if c["op"] == "backward" else 4  # five matrix products of d channels a pair, or two
    return float(products * _sum_mask(c) * c["head_dim"] * c["B"] * c["H"])


# Ranges that the listed cases stand for: operation, data type, sides of the grid, largest number of heads.
_RANGES = [
    ("forward", "bf16", 16, 512, 24),
    ("forward", "bf16", 16, 512, 24),
    ("layer", "bf16", 16, 128, 24),
    ("backward", "bf16", 16, 128, 24),
    ("forward", "f32", 16, 64, 24),
    ("backward", "f32", 8, 40, 24),
    ("forward_host", "bf16", 32, 96, 24),
]


def draw(rng):
    op, dtype, lo, hi, heads = rng.choice(_RANGES)

    def spread(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    def side():
        s = min(hi, max(lo, round(spread(lo, hi))))
        return s if rng.random() < 0.5 else max(lo, s // 8 * 8)  # resolutions are often multiples of 128 pixels

    c = _case("", op, dtype, rng.choice((1, 1, 2)), rng.choice((2, 8, 12, 16, heads)), side(), side(),
              rng.choice((0, 16, 77, 128, 256, 512, rng.randint(1, 512))), rng.choice((64, 128, 128)),
              round(2 * spread(4, 32)) / 2)
    del c["name"]
    most = max(_flops(x) for x in listed() if x["op"] == op and x["dtype"] == dtype)
    while _flops(c) > most:
        key = max(("grid_h", "grid_w"), key=c.get) if c["B"] * c["H"] <= 4 else "B" if c["B"] > 1 else "H"
        c[key] = max(1, c[key] * 3 // 4)
    return c


def prepare(case, seed):
    dev, dtype = torch.device("cuda"), DTYPES[case["dtype"]]
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    B, H, d = case["B"], case["H"], case["head_dim"]
    shape = (B, H, case["n_text"] + case["grid_h"] * case["grid_w"], d)

    def normal(unit_rows=False):
        x = torch.randn(shape, generator=gen, device=dev, dtype=torch.float32)
        if unit_rows:  # as a model's normalisation of Q and K leaves them
            x /= torch.sqrt(x.pow(2).mean(dim=-1, keepdim=True) + 1e-6)
        return x.to(dtype)

    normed = case["dtype"] == "bf16" and case["op"] != "layer"
    s = {"case": case, "op": case["op"], "q": normal(normed), "k": normal(normed), "v": normal(),
         "geometry": (case["grid_h"], case["grid_w"], case["n_text"]), "scale": 1.0 / math.sqrt(d)}
    if case["op"] == "backward":
        s["d_out"] = normal()
        s["dq"], s["dk"], s["dv"] = (torch.empty(shape, device=dev, dtype=dtype) for _ in range(3))
        return s
    s["out"] = torch.empty(shape, device=dev, dtype=dtype)
    if case["op"] == "layer":
        s["q_rot"], s["k_rot"] = torch.empty_like(s["q"]), torch.empty_like(s["k"])
        s["gain_q"], s["gain_k"] = (1.0 + 0.1 * torch.randn(d, generator=gen, device=dev) for _ in range(2))
        s["axes"] = (d // 8, d * 7 // 16, d * 7 // 16)  # (16, 56, 56) of 128 channels
    if case["op"] == "forward_host":
        for name in ("q", "k", "v", "out"):
            s[name] = s[name].cpu().pin_memory()
        s["plan"] = _plan(case)
    return s


_plans = {}


def _plan(c):
    """The plan a program keeps for a shape, whatever its inputs."""
    key = tuple(c[k] for k in ("B", "H", "grid_h", "grid_w", "n_text", "head_dim", "radius"))
    if key not in _plans:
        _plans.clear()
        _plans[key] = clear.Plan(*key)
    return _plans[key]


def run(s):
    gh, gw, T = s["geometry"]
    radius, scale, f32 = s["case"]["radius"], s["scale"], s["case"]["dtype"] == "f32"
    if s["op"] == "forward":
        fwd = clear.clear_attn_fwd_f32 if f32 else clear.clear_attn_fwd
        return fwd(s["q"], s["k"], s["v"], s["out"], gh, gw, T, radius, scale)
    if s["op"] == "layer":
        clear.clear_qk_norm_rope(s["q"], s["k"], s["q_rot"], s["k_rot"], gh, gw, T, s["axes"], s["gain_q"], s["gain_k"])
        out = clear.clear_attn_fwd(s["q_rot"], s["k_rot"], s["v"], s["out"], gh, gw, T, radius, scale)
        return s["q_rot"], s["k_rot"], out
    if s["op"] == "backward":
        bwd = clear.clear_attn_bwd_f32 if f32 else clear.clear_attn_bwd_bf16_tc
        return bwd(s["q"], s["k"], s["v"], s["d_out"], s["dq"], s["dk"], s["dv"], gh, gw, T, radius, scale)
    return s["plan"].forward_host(s["q"], s["k"], s["v"], s["out"], scale)


def work(case):
    tensor = (case["B"] * case["H"] * (case["n_text"] + case["grid_h"] * case["grid_w"]) * case["head_dim"]
              * (2 if case["dtype"] == "bf16" else 4))
    # q, k, v, out; a backward pass reads q, k, v, d_out and writes three gradients; a layer also writes the
    # prepared q and k
    tensors = {"backward": 7, "layer": 6}.get(case["op"], 4)
    return {"bytes": float(tensors * tensor), "flops": _flops(case)}


def tolerance(case):
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
