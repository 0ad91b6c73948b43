"""The work a user of this library has it do, as cases that can be timed and compared.

A case is one pass through the public entry points: the linears of a decoder layer in the launches that a decoder allows
({q, k, v} in one batched call, o, the gated unit over (gate, up), down on the unit's output), one linear alone, a layer whose
activations live in host memory, or a weight matrix materialised.  Sizes are the layer shapes of `synth`, the sizes of the
repository's tests and benchmark, and generic ones; formats are the paper's (W2-G64, W3-G64, W2-G256, W4-G128) and the
benchmark's (K = 2 and 3 at g = 128).  Packed weights come from the library's seeded device generator, activations are N(0, 1) in
binary16, as everywhere in this repository.
"""
import math

import numpy as np
import torch

from paper_2602_04163_b200 import binding, synth

SHAPES = {"7b": {n: (o, i) for n, o, i in synth.QWEN25_7B_LAYER}, "72b": {n: (o, i) for n, o, i in synth.QWEN25_72B_LAYER}}
FORMATS = ((2, 64), (3, 64), (2, 128), (3, 128), (2, 256), (4, 128))
NAMES = ("q", "k", "v", "o", "gate", "up", "down")


def _layer(name, model, K, g, M, **options):
    s = SHAPES[model]
    return dict({"name": name, "kind": "layer", "hidden": s["q"][0], "kv": s["k"][0], "ffn": s["gate"][0], "K": K, "group": g, "M": M,
                 "bias": False, "perm": False}, **options)


def listed():
    return [
        # the smallest call: one token through one 4096 x 4096 linear, where latency counts
        {"name": "linear_4096_1_token", "kind": "linear", "out": 4096, "in": 4096, "K": 2, "group": 128, "M": 1},
        # decoding one sequence with the smaller model (its q, k and v carry a bias): four launches on 69 MB of weights
        _layer("7b_layer_1_token", "7b", 2, 128, 1, bias=True),
        # decoding one sequence with the larger model: 261 MB of weights in four launches
        _layer("72b_layer_1_token", "72b", 2, 128, 1),
        # two sequences (or one with a drafted token) in the paper's W3-G64
        _layer("72b_layer_2_tokens_w3g64", "72b", 3, 64, 2),
        # decoding for a program whose activations live in pinned host memory: x in, one launch over the layer, y out
        _layer("72b_layer_1_token_host", "72b", 3, 128, 1, kind="layer_host"),
        # a few drafted tokens to verify (speculative decoding), an odd number
        _layer("7b_layer_5_tokens", "7b", 3, 128, 5, bias=True),
        # sixteen sequences decoded together
        _layer("72b_layer_16_tokens", "72b", 2, 128, 16),
        # forty-eight sequences decoded together, in the paper's W2-G256 (the down projection's last group is a short one)
        _layer("72b_layer_48_tokens_w2g256", "72b", 2, 256, 48),
        # a short prompt, or a hundred sequences, in the paper's W4-G128
        _layer("7b_layer_100_tokens_w4g128", "7b", 4, 128, 100, bias=True),
        # a prompt of ordinary length, ragged, in W2-G64 with reordered input channels
        _layer("7b_layer_777_tokens_w2g64", "7b", 2, 64, 777, bias=True, perm=True),
        # a long prompt through the larger model: the largest pass
        _layer("72b_layer_4096_tokens", "72b", 3, 128, 4096),
        # the weights of the largest linear rebuilt once, for a caller that multiplies them itself
        {"name": "72b_gate_dequant", "kind": "dequant", "out": 29568, "in": 8192, "K": 2, "group": 128, "M": 1},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("linear", "layer", "layer", "layer", "layer", "layer_host", "dequant"))
    K, g = rng.choice(FORMATS)
    if kind in ("linear", "dequant"):
        out, in_ = 16 * _log_int(rng, 32, 1848), 128 * _log_int(rng, 8, 231)
        if (out // 16) * (in_ // 128) > 1848 * 64:           # no larger than the largest linear of the listed layers
            in_ = 128 * max(8, 1848 * 64 // (out // 16))
        return {"kind": kind, "out": out, "in": in_, "K": K, "group": g, "M": 1 if kind == "dequant" else _log_int(rng, 1, 4096)}
    if rng.random() < 0.4:
        s = SHAPES[rng.choice(("7b", "72b"))]
        hidden, kv, ffn = s["q"][0], s["k"][0], s["gate"][0]
    else:
        hidden, kv, ffn = 128 * _log_int(rng, 8, 64), 16 * _log_int(rng, 16, 64), 128 * _log_int(rng, 24, 231)
    M = rng.choice((1, 1, 2)) if kind == "layer_host" else _log_int(rng, 1, 4096)
    return {"kind": kind, "hidden": hidden, "kv": kv, "ffn": ffn, "K": K, "group": g, "M": M, "bias": rng.random() < 0.5,
            "perm": kind == "layer" and rng.random() < 0.2}


def _linears(case):
    if case["kind"] in ("linear", "dequant"):
        return {"w": (case["out"], case["in"])}
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    return {"q": (h, h), "k": (kv, h), "v": (kv, h), "o": (h, h), "gate": (f, h), "up": (f, h), "down": (h, f)}


def prepare(case, seed):
    M, K, g, kind = case["M"], case["K"], case["group"], case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def acts(n):
        return torch.randn((M, n), generator=gen, device="cuda", dtype=torch.float32).half()

    def buf(n):
        return torch.empty((M, n), device="cuda", dtype=torch.float16)

    lins = _linears(case)
    h = {n: binding.Handle(o, i, K, g, None, (seed << 8) + k, M) for k, (n, (o, i)) in enumerate(lins.items())}
    s = {"kind": kind, "M": M, "h": h}
    if kind == "dequant":
        s["w"] = torch.empty((case["out"], case["in"]), device="cuda", dtype=torch.float16)
        return s
    if kind == "linear":
        s["x"], s["y"] = acts(case["in"]), buf(case["out"])
        return s
    rs = np.random.RandomState(seed % 2 ** 32)
    if case["bias"]:                                         # decoder layers of this kind carry one on q, k and v
        for n in ("q", "k", "v"):
            h[n].bpdq_set_bias(rs.randn(lins[n][0]).astype(np.float16).view(np.uint16))
    if case["perm"]:
        for n in NAMES:
            h[n].bpdq_set_input_permutation(rs.permutation(lins[n][1]).astype(np.int32))
    if kind == "layer_host":                                 # each linear has its own pinned input and output
        s["x"] = [acts(lins[n][1]).cpu().pin_memory() for n in NAMES]
        s["y"] = [torch.empty((M, lins[n][0]), dtype=torch.float16).pin_memory() for n in NAMES]
        s["hs"] = [h[n] for n in NAMES]
        return s
    s["x"], s["attn"], s["mid"] = acts(case["hidden"]), acts(case["hidden"]), acts(case["hidden"])
    for n in ("q", "k", "v", "o", "down"):
        s[n] = buf(lins[n][0])
    s["unit"] = buf(case["ffn"])
    return s


def run(s):
    h, M = s["h"], s["M"]
    stream = torch.cuda.current_stream().cuda_stream
    if s["kind"] == "dequant":
        h["w"].bpdq_dequant(s["w"].data_ptr(), stream)
        return s["w"]
    if s["kind"] == "linear":
        h["w"].bpdq_linear(s["x"].data_ptr(), s["y"].data_ptr(), M, stream)
        return s["y"]
    if s["kind"] == "layer_host":
        binding.bpdq_linear_batch_host(s["hs"], [t.data_ptr() for t in s["x"]], [t.data_ptr() for t in s["y"]], M, stream)
        return s["y"]
    x = s["x"].data_ptr()
    if M <= binding.GEMV_MAX_M:                              # the most tokens a batched call takes
        binding.bpdq_linear_batch([h["q"], h["k"], h["v"]], [x, x, x], [s["q"].data_ptr(), s["k"].data_ptr(), s["v"].data_ptr()], M, stream)
    else:
        for n in ("q", "k", "v"):
            h[n].bpdq_linear(x, s[n].data_ptr(), M, stream)
    h["o"].bpdq_linear(s["attn"].data_ptr(), s["o"].data_ptr(), M, stream)
    binding.bpdq_gate_up_swiglu(h["gate"], h["up"], s["mid"].data_ptr(), s["unit"].data_ptr(), M, stream)
    h["down"].bpdq_linear(s["unit"].data_ptr(), s["down"].data_ptr(), M, stream)
    return {n: s[n] for n in ("q", "k", "v", "o", "unit", "down")}


def work(case):
    """Packed weights once, every activation read once, every output written once; two operations per weight and token."""
    M, K, g, kind = case["M"], case["K"], case["group"], case["kind"]
    lins = _linears(case)
    weights = sum(o * i for o, i in lins.values())
    packed = sum(o * i * K // 8 + o * -(-i // g) * (K + 1) * 2 for o, i in lins.values())
    if kind == "dequant":
        return {"bytes": packed + 2 * weights, "flops": 0}
    if kind == "linear":
        values = case["in"] + case["out"]
    elif kind == "layer_host":
        values = sum(o + i for o, i in lins.values())
    else:                                                    # inputs of {q, k, v}, o and (gate, up); q, k, v, o, the unit, down
        values = 3 * case["hidden"] + 3 * case["hidden"] + 2 * case["kv"] + case["ffn"]
    return {"bytes": packed + 2 * M * values, "flops": 2 * M * weights}


def _s64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _mix(z):
    """splitmix64's output function on int64 tensors (products wrap, shifts are logical)."""
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * _s64(0xBF58476D1CE4E5B9)
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * _s64(0x94D049BB133111EB)
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _draws(seed, tensor, counter):
    golden = 0x9E3779B97F4A7C15
    key = _mix(torch.tensor([_s64((seed ^ (tensor * golden)) & (1 << 64) - 1)], device="cuda"))
    return _mix(key + counter * _s64(golden))


def _weights64(out, in_, K, g, seed, r0, r1):
    """Rows r0..r1-1 of the weights that the seed stands for, in binary64 with nothing rounded: c0 + sum_i ci * bi of the
    seeded planes (one draw per 32 columns) and binary16 coefficients (twelve 16-bit uniforms for c0, one 24-bit uniform else)."""
    r = torch.arange(r0, r1, device="cuda", dtype=torch.int64)[:, None]
    ng, nw = -(-in_ // g), in_ // 32
    group = torch.arange(in_, device="cuda") // g
    bit = torch.arange(32, device="cuda")
    w = None
    for i in range(K + 1):
        e = (i * out + r) * ng + torch.arange(ng, device="cuda")[None, :]
        if i == 0:
            total = torch.zeros_like(e)
            for part in range(3):
                d = _draws(seed, 2, 4 * e + part)
                for q in range(4):
                    total += (d >> (16 * q)) & 0xFFFF
            c = (total - 6 * 65535).float() * (float.fromhex("0x1.47ae14p-6") * 2.0 ** -16)
        else:
            u = ((_draws(seed, 2, 4 * e) >> 40) & 0xFFFFFF).float()
            lo, span = ("0x1.47ae14p-8", "0x1.70a3d8p-5") if i <= 2 else ("0x1.0624dep-9", "0x1.26e978p-6")
            c = u * (float.fromhex(span) * 2.0 ** -24) + float.fromhex(lo)
        c = c.half().double()[:, group]
        if i == 0:
            w = c
        else:
            word = _draws(seed, 1, ((i - 1) * out + r) * nw + torch.arange(nw, device="cuda")[None, :]) >> 32
            w += c * ((word[:, :, None] >> bit) & 1).reshape(r1 - r0, in_)
    return w


def exact(case, seed):
    """run()'s outputs in binary64 from Eq. 1 as it stands (no rounding of weights, sums or the unit).  The rebuilt weights of
    the dequantisation have a definition of their own, bit by bit, and are compared as they are."""
    M, K, g, kind = case["M"], case["K"], case["group"], case["kind"]
    if kind == "dequant":
        return None
    lins = _linears(case)
    seeds = {n: (seed << 8) + k for k, n in enumerate(lins)}
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def acts(n):
        return torch.randn((M, n), generator=gen, device="cuda", dtype=torch.float32).half().double()

    def linear(n, x):
        out, in_ = lins[n]
        return torch.cat([x @ _weights64(out, in_, K, g, seeds[n], r, min(out, r + 2048)).T for r in range(0, out, 2048)], 1)

    if kind == "linear":
        return linear("w", acts(case["in"]))
    rs = np.random.RandomState(seed % 2 ** 32)
    bias, perm = {}, {}
    if case["bias"]:
        bias = {n: torch.from_numpy(rs.randn(lins[n][0]).astype(np.float16)).cuda().double() for n in ("q", "k", "v")}
    if case["perm"]:
        perm = {n: torch.from_numpy(rs.permutation(lins[n][1])).cuda() for n in NAMES}

    def full(n, x):
        y = linear(n, x[:, perm[n]] if n in perm else x)
        return y + bias[n] if n in bias else y

    if kind == "layer_host":
        xs = [acts(lins[n][1]) for n in NAMES]
        return [full(n, x).cpu() for n, x in zip(NAMES, xs)]
    x, attn, mid = acts(case["hidden"]), acts(case["hidden"]), acts(case["hidden"])
    y = {n: full(n, x) for n in ("q", "k", "v")}
    y["o"] = full("o", attn)
    y["unit"] = torch.nn.functional.silu(full("gate", mid)) * full("up", mid)
    y["down"] = full("down", y["unit"])
    return y


def tolerance(case):
    """Rebuilt weights are defined bit by bit.  Everything else: weights may enter the sums rounded to binary16 or unrounded,
    sums may be taken in any order in binary32, outputs are binary16.  Against binary64 sums of the rounded weights the layers'
    outputs are off by up to 5.2e-4 (2-norm) and 0.011 of the root mean square: four times that."""
    return "exact" if case["kind"] == "dequant" else {"rel": 2e-3, "max": 0.05}
