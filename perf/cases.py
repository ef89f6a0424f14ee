"""The measured cases: what a user of this library has it do, through its public entry points.

A video-DiT program calls `vc_attn` once per attention layer and denoising step on the Q, K, V it
has just projected, with a permutation that `vc_group` recomputes every few steps; it may run the
preprocessing pass on its own (the bundle is kept and read by `vc_attn_fwd` later), and it may
hand over host buffers (`vc_attn_host`).  Sizes are the workloads of the benchmark and of the
tests; inputs have their structure: tokens of a smooth field over (t, y, x) plus noise, channel
offsets in K, per-block shifts in V, permutations that gather clusters of value tokens.
"""
import math

import torch

import paper_2609_15810_b200 as vc
from paper_2609_15810_b200 import binding

CLUSTERS = 64            # what the benchmark asks vc_group for

# format -> (bits, p_format, extra flags).  fp8: E4M3 operands and ExpCast-FP8 probabilities (the
# default); int8qk: Q and K as INT8; nvfp4: every operand NVFP4 (the default at 4 bits); hybrid:
# 4-bit storage with ExpCast-FP8 probabilities.
FORMATS = {"fp8": (8, vc.VC_P_DEFAULT, 0), "int8qk": (8, vc.VC_P_DEFAULT, vc.VC_FLAG_INT8_QK),
           "nvfp4": (4, vc.VC_P_DEFAULT, 0), "hybrid": (4, vc.VC_P_EXPCAST_E4M3, 0)}


def _case(call, fmt, B, H, grid, d, perm=True, v_smooth=True, token_major=False, name=None):
    c = {"call": call, "format": fmt, "B": B, "H": H, "t": grid[0], "y": grid[1], "x": grid[2], "d": d,
         "perm": perm, "v_smooth": v_smooth, "token_major": token_major}
    return dict(c, name=name) if name else c


def listed():
    wan = (21, 30, 52)
    return [
        # two heads of a short clip: the smallest call in use, where launches and latency count
        _case("attn", "fp8", 1, 2, (4, 16, 16), 128, name="attn fp8 tiny"),
        # an odd grid, narrow heads, tensors as the projection leaves them ([B, N, H, d]), no permutation
        _case("attn", "fp8", 1, 6, (5, 17, 23), 64, perm=False, token_major=True, name="attn fp8 odd d64"),
        # image-sized sequence of a batch of two, INT8 scores
        _case("attn", "int8qk", 2, 16, (4, 32, 32), 128, name="attn int8qk 4k"),
        # medium clip, narrow heads
        _case("attn", "fp8", 2, 16, (16, 32, 32), 64, name="attn fp8 16k d64"),
        # Wan-1.3B layer on a step behind the grouping window: the permutation at hand, no value smoothing
        _case("attn", "fp8", 1, 12, wan, 128, v_smooth=False, name="attn fp8 wan1.3b frozen"),
        # the same layer with everything, probabilities included, in NVFP4
        _case("attn", "nvfp4", 1, 12, wan, 128, name="attn nvfp4 wan1.3b"),
        # Wan-14B layer, 8 bits: the headline workload
        _case("attn", "fp8", 1, 40, wan, 128, name="attn fp8 wan14b"),
        # ... and in the hybrid 4-bit arrangement
        _case("attn", "hybrid", 1, 40, wan, 128, name="attn hybrid wan14b"),
        # HunyuanVideo-sized sequence: the largest call
        _case("attn", "hybrid", 1, 24, (33, 45, 80), 128, name="attn hybrid hunyuan"),
        # the preprocessing pass on its own
        _case("prep", "fp8", 1, 40, wan, 128, name="prep fp8 wan14b"),
        # warm-started regrouping of a step's values
        _case("group", "fp8", 1, 40, wan, 128, perm=False, name="group wan14b"),
        # host buffers in, host buffer out
        _case("host", "fp8", 1, 12, wan, 128, name="host fp8 wan1.3b"),
    ]


def _flops(c):
    n = c["t"] * c["y"] * c["x"]
    return 4.0 * c["B"] * c["H"] * n * n * c["d"]


_MOST = _flops(_case("attn", "hybrid", 1, 24, (33, 45, 80), 128))


def draw(rng):
    """Any entry point, format and layout; sequences of 200 to 118800 tokens on odd and even grids."""
    while True:
        call = rng.choice(["attn"] * 6 + ["prep", "prep_stats", "group", "host"])
        fmt = rng.choice(["fp8", "fp8", "nvfp4", "hybrid", "int8qk"])
        if call == "prep_stats" and fmt not in ("fp8", "int8qk"):
            fmt = "fp8"          # supplied statistics are an 8-bit entry point
        d = rng.choice([128, 128, 64])
        n = math.exp(rng.uniform(math.log(200), math.log(118800)))
        t = rng.randint(1, 33)
        x = max(1, round(math.sqrt(n / t) * rng.uniform(0.8, 1.6)))
        y = max(1, round(n / t / x))
        B = rng.choice([1, 1, 2])
        H = rng.choice([1, 2, 3, 6, 12, 16, 24, 40])
        c = _case(call, fmt, B, H, (t, y, x), d, perm=call != "group" and rng.random() < 0.75,
                  v_smooth=rng.random() < 0.75, token_major=call not in ("host", "prep_stats") and rng.random() < 0.3)
        n = t * y * x
        # (NVFP4 probabilities, INT8 scores and narrow heads cost more per product)
        most = (0.2 if fmt in ("nvfp4", "int8qk") else 0.6) * _MOST * (d / 128)
        if n < CLUSTERS or n > 118800 or B * H * n > 40 * 118800 or _flops(c) > most:
            continue
        if call == "host" and B * H * n > 40 * 32760:
            continue
        return c


# ----------------------------------------------------------------------------- inputs
def _inputs(c, seed):
    """Q, K, V as [B, H, N, d] bf16 on the GPU (views of [B, N, H, d] memory with token_major)."""
    B, H, d = c["B"], c["H"], c["d"]
    T, Y, X = c["t"], c["y"], c["x"]
    N = T * Y * X
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = torch.arange(N, device="cuda")
    pos = torch.stack([(n // (Y * X)) / T, (n // X) % Y / Y, n % X / X], dim=1).float()
    nb = (N + 127) // 128
    out = []
    for tensor in range(3):
        if c["token_major"]:
            full = torch.empty(B, N, H, d, dtype=torch.bfloat16, device="cuda").transpose(1, 2)
        else:
            full = torch.empty(B, H, N, d, dtype=torch.bfloat16, device="cuda")
        for b in range(B):
            for h in range(H):
                a = 0.5 * torch.randn(N, d, generator=g, device="cuda")
                f = 4.0 * math.pi * torch.rand(8, 3, d, generator=g, device="cuda")
                phase = 2.0 * math.pi * torch.rand(8, 1, d, generator=g, device="cuda")
                for k in range(8):                   # unit variance: eight waves of amplitude 1/2
                    a.add_(torch.addmm(phase[k], pos, f[k]).sin_(), alpha=0.5)
                if tensor == 1:
                    a += 3.0 * torch.randn(1, d, generator=g, device="cuda")
                if tensor == 2:
                    a += torch.randn(nb, d, generator=g, device="cuda").repeat_interleave(128, dim=0)[:N]
                full[b, h] = a
        out.append(full)
    return out, g


def _cluster_perm(v, g):
    """Tokens sorted by the nearest of 64 random directions: contiguous runs of similar value rows."""
    B, H, N, d = v.shape
    perm = torch.empty(B, H, N, dtype=torch.int32, device="cuda")
    dirs = torch.randn(d, CLUSTERS, generator=g, device="cuda")
    for b in range(B):
        for h in range(H):
            perm[b, h] = torch.argsort((v[b, h].float() @ dirs).argmax(dim=1), stable=True)
    return perm


def prepare(case, seed):
    (q, k, v), g = _inputs(case, seed)
    B, H, N, d = v.shape
    bits, p_format, flags = FORMATS[case["format"]]
    flags |= vc.VC_FLAG_ALL if case["v_smooth"] else vc.VC_FLAG_ALL & ~vc.VC_FLAG_V_SMOOTH
    strides = {"stride_b": v.stride(0), "stride_h": v.stride(1), "stride_n": v.stride(2)} if case["token_major"] else {}
    p = vc.Params.make(B, H, N, d, (case["t"], case["y"], case["x"]), bits=bits, p_format=p_format, flags=flags, **strides)
    s = {"call": case["call"], "bits": bits, "p": p, "q": q, "k": k, "v": v,
         "perm": _cluster_perm(v, g) if case["perm"] else None}
    if case["call"] == "group":
        # centroids as an earlier step left them: rows of V with this step's noise on top
        rows = torch.arange(CLUSTERS, device="cuda") * (N // CLUSTERS)
        s["centroids"] = (v[:, :, rows].float() + 0.1 * torch.randn(B, H, CLUSTERS, d, generator=g, device="cuda")).contiguous()
        s["perm"] = torch.empty(B, H, N, dtype=torch.int32, device="cuda")
        s["work"] = torch.empty(vc.vc_group_workspace_bytes(p), dtype=torch.uint8, device="cuda")
        del s["q"], s["k"]
        return s
    s["quant"], s["work"] = binding.alloc_buffers(p)
    s["o"] = torch.empty(B, H, N, d, dtype=torch.bfloat16, device="cuda")
    if case["call"] == "host":
        s["host"] = [t.cpu().pin_memory() if t is not None else None for t in (q, k, v, s["perm"])]
        s["o_host"] = torch.empty(B, H, N, d, dtype=torch.bfloat16, pin_memory=True)
    if case["call"] == "prep_stats":
        s["stats"] = _statistics(case, k, v, s["perm"])
    if case["call"] in ("prep", "prep_stats"):
        s["bundle"] = _bundle(s)
    return s


def _statistics(case, k, v, perm):
    """What a producer of K and V hands over: the rotated K's channel mean, V's block means and residual maxima."""
    B, H, N, d = v.shape
    side = 2 * (d // 6)
    dims = (d - 2 * side, side, side)
    n = torch.arange(N, device="cuda")
    pos = (n // (case["y"] * case["x"]), (n // case["x"]) % case["y"], n % case["x"])
    phi = torch.cat([pos[a].double()[:, None] * 10000.0 ** (-torch.arange(0, dims[a], 2, device="cuda").double() / dims[a])
                     for a in range(3)], dim=1)
    cos, sin = phi.cos().float(), phi.sin().float()
    nb = (N + 127) // 128
    mean = torch.empty(B * H, d, device="cuda")
    mu = torch.zeros(B * H, nb, d, device="cuda")
    amax = torch.empty(B * H, d, device="cuda")
    for bh in range(B * H):
        x = k[bh // H, bh % H].float()
        x0, x1 = x[:, 0::2], x[:, 1::2]
        mean[bh] = torch.stack([x0 * cos - x1 * sin, x0 * sin + x1 * cos], dim=2).reshape(N, d).double().mean(dim=0).float()
        w = v[bh // H, bh % H].float()
        if perm is not None:
            w = w[perm[bh // H, bh % H].long()]
        if case["v_smooth"]:
            pad = torch.zeros(nb * 128, d, device="cuda")
            pad[:N] = w
            count = torch.full((nb, 1), 128.0, device="cuda")
            count[-1] = N - 128 * (nb - 1)
            mu[bh] = pad.view(nb, 128, d).sum(dim=1) / count
        amax[bh] = (w - mu[bh].repeat_interleave(128, dim=0)[:N]).abs().amax(dim=0)
    return mean, mu, amax


def _bundle(s):
    """The sections of the quantized bundle that the pass writes, as tensors."""
    view = vc.vc_quant_view(s["p"], s["quant"])
    names = ["q_codes", "k_codes", "v_codes", "q_scale", "k_scale", "v_scale", "v_means", "k_mean"]
    if s["bits"] == 4:
        names += ["q_micro", "k_micro", "v_micro"]
    kind = {"q_scale": torch.float32, "k_scale": torch.float32, "v_scale": torch.float32, "v_means": torch.bfloat16,
            "k_mean": torch.float32}
    return {n: binding.section(view, n, s["quant"], kind.get(n, torch.uint8)) for n in names}


# ----------------------------------------------------------------------------- one pass
def run(s):
    p = s["p"]
    if s["call"] == "attn":
        vc.vc_attn(p, s["q"], s["k"], s["v"], s["perm"], s["o"], s["quant"], s["work"])
        return s["o"]
    if s["call"] == "prep":
        vc.vc_prep(p, s["q"], s["k"], s["v"], s["perm"], s["quant"], s["work"])
        return s["bundle"]
    if s["call"] == "prep_stats":
        vc.vc_prep_with_stats(p, s["q"], s["k"], s["v"], s["perm"], *s["stats"], s["quant"], s["work"])
        return s["bundle"]
    if s["call"] == "group":
        vc.vc_group(p, s["v"], CLUSTERS, 1, True, s["centroids"], s["perm"], s["work"])
        return {"perm": s["perm"], "centroids": s["centroids"]}
    q, k, v, perm = s["host"]
    vc.vc_attn_host(p, q, k, v, perm, s["o_host"], s["q"], s["k"], s["v"], s["perm"], s["o"], s["quant"], s["work"])
    return s["o_host"]


def work(case):
    """Inputs read once, outputs written once; the products of the path."""
    B, H, d = case["B"], case["H"], case["d"]
    N = case["t"] * case["y"] * case["x"]
    n_pad = 128 * ((N + 127) // 128)
    row = float(B * H * N)
    bits = FORMATS[case["format"]][0]
    perm = 4.0 * row if case["perm"] else 0.0
    if case["call"] == "group":
        return {"bytes": 2 * row * d + 4 * row + 8.0 * B * H * CLUSTERS * d, "flops": 4 * row * CLUSTERS * d}
    if case["call"] in ("prep", "prep_stats"):
        codes = B * H * n_pad * d * 3 * (1.0 if bits == 8 else 0.5625)
        rest = B * H * d * (n_pad // 128) * 2.0
        if case["call"] == "prep_stats":
            rest += B * H * d * ((n_pad // 128) * 4.0 + 8.0)
        return {"bytes": 6 * row * d + perm + codes + rest, "flops": 2 * row * d * (6 + math.log2(d) * 2)}
    return {"bytes": 8 * row * d + perm, "flops": _flops(case)}


def tolerance(case):
    # Each about four times the largest distance between this library and the emulation of the same
    # quantized path in 64 bits (1955 to 32760 tokens, every format): outputs 5.7e-4 and 0.011 (a
    # bf16 step is 2^-8, and a score on the edge of two probability codes falls either way);
    # bundles 1.9e-5 of the codes one step apart, scales and means 5.7e-8 and 2.2e-7 except for a
    # block mean, which may round to the next bf16 value; centroids 4.8e-8 and 4.4e-7, labels the same.
    if case["call"] == "group":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-4}
    if case["call"] in ("prep", "prep_stats"):
        return {"rel": 1e-4, "max": 4e-3, "differ": 1e-4}
    return {"rel": 2.5e-3, "max": 0.045}
