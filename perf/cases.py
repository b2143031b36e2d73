"""The work that programs using this package have it do, as measurable cases.

A serving process holds one packed head and runs its forward on the hidden
states of the current step: one token or a handful per step (latency, memory
bound), tens to hundreds of tokens (large decode batches, verification of
drafted tokens, prompt chunks), or thousands (prefill, perplexity scoring).
It asks for logits, the greedy token or the cross entropy of given targets.
Offline, a head is constructed: dense factors and residuals are quantised,
packed and dequantised again.

Heads are drawn on the GPU in the canonical packed layout (uniform codes, fp16
scales with a full mantissa) and hidden states are anisotropic with a few
outlier channels, as in the package's synthetic inputs.
"""

import math

import torch

from paper_2608_02703_gb300 import archead, construct

# Element rms of the head's parts (logits come out with rms near 2 at d = 4096).
_RMS_RESIDUAL, _RMS_CORE, _RMS_CORR = 0.004, 0.008, 0.0012


class _Shape:
    """Head shape as archead_pack_create takes it."""

    def __init__(self, case):
        self.V, self.d = case["V"], case["d"]
        self.core_rank, self.corr_rank, self.group_size = case["rc"], case["rr"], case["g"]
        self.fmt = case["fmt"]


def _case(op, V, d, rc, rr, g, fmt, M, out="bf16"):
    return dict(op=op, V=V, d=d, rc=rc, rr=rr, g=g, fmt=fmt, M=M, out=out)


_QWEN = dict(V=151936, d=4096, rc=128, rr=32, g=128, fmt="int8")       # Qwen3-8B-shaped head, INT8 format
_QWEN_SC4 = dict(V=151936, d=4096, rc=10, rr=6, g=64, fmt="sc4")       # the same in the paper's packed format
_GEMMA = dict(V=262144, d=2560, rc=128, rr=32, g=128, fmt="int8")      # Gemma-4-E4B-shaped head
_TINY = dict(V=4096, d=512, rc=64, rr=16, g=64, fmt="int8")            # small head: latency only


def listed():
    named = [
        # A small model's step: everything fits in cache, launches and latency count.
        ("tiny head, 4 tokens", _case("logits", M=4, **_TINY)),
        # One user generating: sampling needs the whole logits row.
        ("decode 1 token", _case("logits", M=1, **_QWEN)),
        # One user generating greedily on a head in the paper's format.
        ("greedy 1 token, paper format", _case("argmax", M=1, **_QWEN_SC4)),
        # A small serving batch of odd size; the sampler takes fp32 logits.
        ("decode 13 tokens, wide vocabulary", _case("logits", M=13, out="fp32", **_GEMMA)),
        # Serving batches.
        ("decode 24 tokens", _case("logits", M=24, **_QWEN)),
        ("decode 64 tokens", _case("logits", M=64, **_QWEN)),
        # A ragged prompt chunk or drafted tokens of several users being verified.
        ("verify 200 tokens, paper format", _case("logits", M=200, **_QWEN_SC4)),
        # Scoring one passage: cross entropy per token, no logits written.
        ("score 512 tokens, wide vocabulary", _case("ce", M=512, **_GEMMA)),
        # Perplexity over a long window.
        ("score 2048 tokens, paper format", _case("ce", M=2048, **_QWEN_SC4)),
        # Prefill with all logits (the largest call).
        ("prefill 4096 tokens", _case("logits", M=4096, **_QWEN)),
        # Offline construction: the residual in the paper's format, quantised and packed.
        ("construct residual, paper format", _case("residual_sc4", M=0, **_QWEN_SC4)),
        # Offline construction, INT8 format: core factor per column, residual per group, realized residual.
        ("construct INT8 parts", _case("quantize_int8", M=0, V=151936, d=1024, rc=128, rr=32, g=128, fmt="int8")),
    ]
    return [dict(c, name=n) for n, c in named]


def draw(rng):
    """One more case: sizes spread over the ranges the package serves."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["logits", "logits", "logits", "argmax", "ce", "ce", "residual_sc4", "quantize_int8"])
    fmt = rng.choice(["int8", "sc4"])
    if op == "residual_sc4":
        fmt = "sc4"
    if op == "quantize_int8":
        fmt = "int8"
    g = rng.choice([32, 64, 128, 128, 256])
    unit = max(g, 64)
    d = unit * max(1, log_int(256, 6144) // unit)
    V = log_int(1000, 262144)
    if fmt == "sc4":
        rc, rr = rng.randint(4, 32), rng.randint(2, 16)
    else:
        rc, rr = rng.choice([0, 16, 33, 64, 128, 200]), rng.choice([0, 8, 16, 32, 48])
    if op in ("residual_sc4", "quantize_int8"):
        while V * d > 151936 * 4096:
            V //= 2
        return _case(op, V, d, max(rc, 1), rr, g, fmt, 0)
    M = log_int(1, 4096)
    while M > 1 and M * V * d > 4096 * 151936 * 4096:
        M //= 2
    return _case(op, V, d, rc, rr, g, fmt, M, out=rng.choice(["bf16", "bf16", "fp32"]))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _scales(gen, base, shape):
    """fp16 scales base * 2^U(-1/2, 1/2)."""
    u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32) - 0.5
    return (base * torch.exp2(u)).to(torch.float16)


def _codes(gen, lo, hi, shape):
    return torch.randint(lo, hi, shape, generator=gen, device="cuda", dtype=torch.int8)


def _pack5(codes):
    """5-bit two's complement codes as each row's little-endian bit string."""
    V, r = codes.shape
    nb = (5 * r + 7) // 8
    bits = torch.zeros((V, 8 * nb), dtype=torch.uint8, device=codes.device)
    for b in range(5):
        bits[:, b:5 * r:5] = ((codes >> b) & 1).to(torch.uint8)
    w = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.int32, device=codes.device)
    return (bits.view(V, nb, 8).to(torch.int32) * w).sum(-1).to(torch.uint8)


def _head(case, gen):
    """Canonical packed arrays, plus the core codes as int8 ("u")."""
    V, d, rc, rr, g = case["V"], case["d"], case["rc"], case["rr"], case["g"]
    G = d // g
    sc4 = case["fmt"] == "sc4"
    rms4 = math.sqrt(sum(c * c for c in range(-8, 8)) / 16)
    ms8 = sum(c * c for c in range(-127, 128)) / 255
    ms5 = sum(c * c for c in range(-16, 16)) / 32
    base_c = math.sqrt(_RMS_CORE / (math.sqrt(max(rc, 1)) * ms8))
    base_w = math.sqrt(_RMS_CORR / (math.sqrt(max(rr, 1)) * ms8))
    h = {"res_codes": torch.randint(0, 256, (V, d // 2), generator=gen, device="cuda", dtype=torch.uint8)}
    if sc4:
        rms_q = math.sqrt(sum(q * q for q in range(1, 17)) / 16)
        q = torch.randint(0, 256, (V, (G + 1) // 2), generator=gen, device="cuda", dtype=torch.uint8)
        if G % 2:
            q[:, -1] &= 15
        h["res_scale_codes"] = q
        h["res_row_scale"] = _scales(gen, _RMS_RESIDUAL / rms4 / rms_q, (V,))
        u = _codes(gen, -16, 16, (V, rc))
        h["core_u5"] = _pack5(u)
        h["core_u_scale"] = _scales(gen, base_c * math.sqrt(ms8 / ms5), (rc,))
    else:
        h["res_scales"] = _scales(gen, _RMS_RESIDUAL / rms4, (V, G))
        u = _codes(gen, -127, 128, (V, rc))
        h["core_u"] = u
        h["core_u_scale"] = _scales(gen, base_c, (rc,))
    h["core_v"] = _codes(gen, -127, 128, (d, rc))
    h["core_v_scale"] = _scales(gen, base_c, (rc,))
    h["corr_a"] = _codes(gen, -127, 128, (V, rr))
    h["corr_a_scale"] = _scales(gen, base_w, (V,))
    h["corr_b"] = _codes(gen, -127, 128, (d, rr))
    h["corr_b_scale"] = _scales(gen, base_w, (G, rr))
    return h, u


def _hidden(case, gen):
    """Anisotropic hidden states with four outlier channels, bf16 [M, d]."""
    M, d = case["M"], case["d"]
    x = torch.randn((M, d), generator=gen, device="cuda") * torch.logspace(-2.0, 1.0, d, device="cuda")
    for _ in range(3):  # rotate by Householder reflections
        v = torch.randn((d,), generator=gen, device="cuda")
        v /= v.norm()
        x -= 2.0 * (x @ v)[:, None] * v[None, :]
    x[:, torch.randint(0, d, (4,), generator=gen, device="cuda")] *= 20.0
    return x.to(torch.bfloat16).contiguous()


def _targets(case, gen):
    return torch.randint(0, case["V"], (case["M"],), generator=gen, device="cuda", dtype=torch.int32)


def _dense(case, gen):
    """A dense residual: Gaussian with a row-dependent size."""
    size = _RMS_RESIDUAL * torch.exp2(torch.rand((case["V"], 1), generator=gen, device="cuda") * 2 - 1)
    return torch.randn((case["V"], case["d"]), generator=gen, device="cuda") * size


def _factor(case, gen):
    return torch.randn((case["V"], case["rc"]), generator=gen, device="cuda") * 0.1


def prepare(case, seed):
    gen = _gen(seed)
    s = {"op": case["op"], "g": case["g"], "M": case["M"]}
    V, d, M = case["V"], case["d"], case["M"]
    if case["op"] == "residual_sc4":
        s["r"] = _dense(case, gen)
        return s
    if case["op"] == "quantize_int8":
        s["r"], s["f"] = _dense(case, gen), _factor(case, gen)
        return s
    head, _ = _head(case, gen)
    s["pack"] = archead.archead_pack_create(head, _Shape(case))
    s["x"] = _hidden(case, gen)
    if case["op"] == "logits":
        fp32 = case["out"] == "fp32"
        s["dtype"] = archead.OUT_FP32 if fp32 else archead.OUT_BF16
        s["y"] = torch.empty((M, V), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    elif case["op"] == "argmax":
        s["index"] = torch.empty((M,), dtype=torch.int32, device="cuda")
        s["value"] = torch.empty((M,), dtype=torch.float32, device="cuda")
    else:
        s["targets"] = _targets(case, gen)
        s["ce"] = torch.empty((M,), dtype=torch.float32, device="cuda")
    return s


def run(s):
    if s["op"] == "logits":
        archead.archead_forward(s["pack"], s["x"], s["M"], s["y"], s["dtype"])
        return s["y"]
    if s["op"] == "argmax":
        archead.archead_forward_argmax(s["pack"], s["x"], s["M"], s["index"], s["value"])
        return {"index": s["index"], "value": s["value"]}
    if s["op"] == "ce":
        archead.archead_forward_ce(s["pack"], s["x"], s["M"], s["targets"], s["ce"])
        return s["ce"]
    if s["op"] == "residual_sc4":
        r, g = s["r"], s["g"]
        rows, cols = r.shape
        codes = torch.empty((rows, cols), dtype=torch.int8, device="cuda")
        scale_codes = torch.empty((rows, cols // g), dtype=torch.uint8, device="cuda")
        row_scale = torch.empty((rows,), dtype=torch.int16, device="cuda")
        archead.archead_quantize_residual_sc4(r, g, codes, scale_codes, row_scale)
        return {"codes": construct.pack(codes, 4), "scale_codes": construct.pack(scale_codes.view(torch.int8), 4),
                "row_scale": row_scale}
    u, us = construct.quantize(s["f"], s["f"].shape[0], 1, 8)
    r, rs = construct.quantize(s["r"], 1, s["g"], 4)
    return {"core": u, "core_scale": us, "codes": construct.pack(r, 4), "scales": rs,
            "residual": construct.dequantize(r, rs, 1, s["g"])}


def work(case):
    V, d, rc, rr, g, M = (case[k] for k in ("V", "d", "rc", "rr", "g", "M"))
    G = d // g
    if case["op"] == "residual_sc4":
        return {"bytes": 4 * V * d + V * d // 2 + V * ((G + 1) // 2) + 2 * V, "flops": 3 * V * d}
    if case["op"] == "quantize_int8":
        return {"bytes": 5 * V * rc + 2 * rc + 4 * V * d + V * d // 2 + 2 * V * G + 4 * V * d, "flops": 4 * V * d}
    if case["fmt"] == "sc4":
        head = V * d // 2 + V * ((G + 1) // 2) + 2 * V + V * ((5 * rc + 7) // 8)
    else:
        head = V * d // 2 + 2 * V * G + V * rc
    head += 4 * rc + d * rc + V * rr + (2 * V if rr else 0) + d * rr + 2 * G * rr
    out = {"logits": M * V * (4 if case["out"] == "fp32" else 2), "argmax": 8 * M, "ce": 8 * M}[case["op"]]
    return {"bytes": head + 2 * M * d + out, "flops": 2 * M * V * d + 2 * M * (V + d) * (rc + rr)}


def tolerance(case):
    if case["op"] in ("residual_sc4", "quantize_int8"):
        return "exact"  # integer decisions in fp32, and code * scale exact in fp32
    if case["op"] == "logits" and case["out"] == "bf16":
        return {"rel": 2e-3}  # one rounding to bf16: sums in another order flip some by one unit
    return {"rel": 4e-5}  # fp32 sums in another order


def _logit_blocks(case, seed):
    """(first row, float64 logits [M, rows], ...) of row blocks, from the definition of the packed head."""
    gen = _gen(seed)
    h, u = _head(case, gen)
    x = _hidden(case, gen).double()
    V, d, rc, rr, g = (case[k] for k in ("V", "d", "rc", "rr", "g"))
    G = d // g
    tc = (x @ h["core_v"].double()) * h["core_v_scale"].double() * h["core_u_scale"].double()
    B = h["corr_b"].double() * h["corr_b_scale"].double().repeat_interleave(g, dim=0)
    tr = x @ B
    step = max(1, (1 << 27) // max(d, case["M"]))

    def blocks():
        for r0 in range(0, V, step):
            r1 = min(V, r0 + step)
            b = h["res_codes"][r0:r1]
            w = torch.stack([b & 15, b >> 4], dim=-1).view(r1 - r0, d).to(torch.float64)
            w = torch.where(w > 7, w - 16, w)
            if case["fmt"] == "sc4":
                q = h["res_scale_codes"][r0:r1]
                q = torch.stack([q & 15, q >> 4], dim=-1).view(r1 - r0, -1)[:, :G].double() + 1
                sc = q * h["res_row_scale"][r0:r1].double()[:, None]
            else:
                sc = h["res_scales"][r0:r1].double()
            w = (w.view(r1 - r0, G, g) * sc[:, :, None]).view(r1 - r0, d)
            y = x @ w.T
            if rc:
                y += tc @ u[r0:r1].double().T
            if rr:
                y += tr @ (h["corr_a"][r0:r1].double() * h["corr_a_scale"][r0:r1].double()[:, None]).T
            yield r0, y

    return gen, blocks()


def exact(case, seed):
    op, V, d, g = case["op"], case["V"], case["d"], case["g"]
    if op in ("residual_sc4", "quantize_int8"):
        return None  # whole numbers decided in fp32; nothing to hold against 64 bits
    if case["M"] * V * d > 3e12 and op != "logits":
        return None
    gen, blocks = _logit_blocks(case, seed)
    if op == "logits":
        y = torch.empty((case["M"], V), dtype=torch.float64, device="cuda")
        for r0, b in blocks:
            y[:, r0:r0 + b.shape[1]] = b
        return y
    if op == "argmax":
        best = torch.full((case["M"],), -math.inf, dtype=torch.float64, device="cuda")
        index = torch.zeros((case["M"],), dtype=torch.int32, device="cuda")
        for r0, b in blocks:
            v, i = b.max(dim=1)
            index = torch.where(v > best, (i + r0).to(torch.int32), index)
            best = torch.maximum(best, v)
        return {"index": index, "value": best}
    t = _targets(case, gen).long()
    lse = torch.full((case["M"],), -math.inf, dtype=torch.float64, device="cuda")
    yt = torch.zeros((case["M"],), dtype=torch.float64, device="cuda")
    for r0, b in blocks:
        lse = torch.logaddexp(lse, torch.logsumexp(b, dim=1))
        here = (t >= r0) & (t < r0 + b.shape[1])
        rows = torch.nonzero(here).squeeze(1)
        yt[rows] = b[rows, t[rows] - r0]
    return lse - yt
