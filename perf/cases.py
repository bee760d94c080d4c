"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is a plain dict; ``prepare`` makes what a program holds before the call (activations, weights packed
once offline, output and workspace buffers), ``run`` is one pass through the public binding, as a program
calls it.  Six kinds:

  linear    the W4A4 layer on packed weights: ``bro.linear``, or ``bro.linear_rs`` with a random sign vector;
            with fp32 output (partial sums that are added up later) ``rotate_quantize_mxfp4`` + ``gemm_mxfp4``
  mlp       the layer behind the gated activation: ``bro.swiglu_linear`` (down_proj with its online rotation)
  stack     one transformer block's linears in a row on the same few tokens: fused qkv, output projection,
            fused gate/up, down projection behind the gated activation
  quantize  rotate + quantise alone, online activations or offline weights, any rotation size and scale layout
  formats   the format study: simulated quantisation of one tensor in every compared 4-bit format
  scales    the scale study: outlier groups, scale bytes before and after the rotation, inflation, group error

Inputs follow the recipe of ``paper_2511_04214_b200.synth`` (Gaussian activations, 1 % of the channels scaled
by Laplace(0, 50), 0.1 % of the tokens by 20; Gaussian weights of deviation 0.02), drawn on the GPU.
"""
import math

import torch

from paper_2511_04214_b200 import binding as bro

STUDY_FORMATS = ("mxfp4", "bfp4", "mxint4", "bint4", "int4_row_asym")
MOST_MACS = 8192 * 8192 * 28672
MOST_ELEMENTS = 16384 * 4096


def listed():
    return [
        # the smallest call: one small layer on 64 tokens, where the latency of a call is all there is
        {"name": "linear-64x2048x2048", "kind": "linear", "M": 64, "K": 2048, "N": 2048, "block": 32, "signs": False, "out": "bf16"},
        # decoding one sequence through a large layer: 125 MB of packed weights for one token
        {"name": "decode-1x8192x28672", "kind": "linear", "M": 1, "K": 8192, "N": 28672, "block": 32, "signs": False, "out": "bf16"},
        # decoding 16 sequences through the four linears of an 8B-shaped block: one token step of a server
        {"name": "decode-block-16", "kind": "stack", "M": 16, "d": 4096, "kv": 1024, "f": 14336, "block": 32},
        # ordinary prefill of a 1B-shaped model
        {"name": "prefill-2048x2048x8192", "kind": "linear", "M": 2048, "K": 2048, "N": 8192, "block": 32, "signs": False, "out": "bf16"},
        # nothing divides: ragged tokens, channels and outputs, the randomised rotation, fp32 partial sums
        {"name": "ragged-777x4384x6004-f32", "kind": "linear", "M": 777, "K": 4384, "N": 6004, "block": 32, "signs": True, "out": "f32"},
        # the layer the paper rotates online: down_proj of an 8B-shaped model on 4096 tokens
        {"name": "mlp-4096x14336x4096", "kind": "mlp", "M": 4096, "K": 14336, "N": 4096, "block": 32},
        # the largest call: prefill of a 70B-shaped layer
        {"name": "prefill-8192x8192x28672", "kind": "linear", "M": 8192, "K": 8192, "N": 28672, "block": 32, "signs": False, "out": "bf16"},
        # packing a layer's weights for the default rotation (offline, and whenever weights change)
        {"name": "pack-14336x4096-b32", "kind": "quantize", "M": 14336, "K": 4096, "block": 32, "signs": False, "layout": "gemm", "weights": True},
        # the rotation sizes above the group, on the activation tensor of the block-size sweep
        {"name": "quantize-16384x4096-b128", "kind": "quantize", "M": 16384, "K": 4096, "block": 128, "signs": False, "layout": "gemm", "weights": False},
        {"name": "quantize-16384x4096-global", "kind": "quantize", "M": 16384, "K": 4096, "block": 0, "signs": False, "layout": "gemm", "weights": False},
        # the two studies of the paper on one activation tensor
        {"name": "formats-8192x4096-b32", "kind": "formats", "M": 8192, "K": 4096, "block": 32},
        {"name": "scales-16384x4096-b32", "kind": "scales", "M": 16384, "K": 4096, "block": 32},
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(max(int(round(v / multiple)) * multiple, multiple, lo), hi)


def _blocks_of(K, sizes):
    return [b for b in sizes if b == 0 and K & (K - 1) == 0 and K <= 32768 or b > 0 and K % b == 0]


def draw(rng):
    kind = rng.choices(("linear", "mlp", "stack", "quantize", "formats", "scales"), (8, 3, 3, 4, 2, 2))[0]
    if kind in ("linear", "mlp"):
        # layers of 1B- to 70B-shaped models, whole or split over GPUs; tokens from decode to long prefill
        K = _log_int(rng, 1024, 14336, 32) if rng.random() < 0.5 else rng.choice((1024, 2048, 4096, 5120, 8192, 11008, 14336))
        N = _log_int(rng, 1024, 28672) if rng.random() < 0.5 else rng.choice((1024, 2048, 4096, 8192, 14336, 28672))
        M = _log_int(rng, 1, 8192) if rng.random() < 0.6 else 1 << rng.randrange(0, 14)
        M = max(1, min(M, MOST_MACS // (K * N)))
        case = {"kind": kind, "M": M, "K": K, "N": N, "block": 32}
        if kind == "linear":
            case["block"] = rng.choice(_blocks_of(K, (32, 32, 32, 32, 64, 128)))
            case["signs"] = rng.random() < 0.25
            case["out"] = "f32" if rng.random() < 0.2 else "bf16"
        return case
    if kind == "stack":
        d = rng.choice((2048, 3072, 4096, 5120, 8192))
        return {"kind": kind, "M": _log_int(rng, 1, 128), "d": d, "kv": d // rng.choice((1, 4, 8)), "f": _log_int(rng, 2 * d, min(4 * d, 14336), 32), "block": 32}
    global_k = kind != "formats" and rng.random() < 0.3
    K = 1 << rng.randrange(10, 15) if global_k else _log_int(rng, 1024, 14336, 32)
    M = _log_int(rng, 16, 16384)
    M = max(1, min(M, MOST_ELEMENTS // (2 if kind == "formats" else 1) // K))
    if kind == "quantize":
        block = 0 if global_k else rng.choice(_blocks_of(K, (16, 32, 32, 64, 64, 128, 128)))
        weights = rng.random() < 0.4
        return {"kind": kind, "M": M, "K": K, "block": block, "signs": rng.random() < 0.25,
                "layout": "gemm" if weights or rng.random() < 0.7 else "canonical", "weights": weights}
    return {"kind": kind, "M": M, "K": K, "block": 0 if global_k else rng.choice(_blocks_of(K, (32, 32, 64, 128)))}


# ---- inputs ----------------------------------------------------------------------------------------------
def _activations(M, K, gen):
    x = torch.randn(M, K, generator=gen, device="cuda", dtype=torch.float32)
    n = max(1, round(0.01 * K))
    cols = torch.randperm(K, generator=gen, device="cuda")[:n]
    u = (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) - 0.5).clamp(-0.5 + 1e-12, 0.5 - 1e-12)
    x[:, cols] *= (-50.0 * torch.sign(u) * torch.log1p(-2.0 * u.abs())).float()
    if M >= 500:
        x[torch.randperm(M, generator=gen, device="cuda")[:int(0.001 * M + 0.5)]] *= 20.0
    return x.to(torch.bfloat16)


def _weights(N, K, gen):
    return (torch.randn(N, K, generator=gen, device="cuda", dtype=torch.float32) * 0.02).to(torch.bfloat16)


def _signs(K, gen):
    return (1 - 2 * torch.randint(0, 2, (K,), generator=gen, device="cuda")).to(torch.bfloat16)


class _Layer:
    """Packed weights with the output and workspace buffers that a program keeps for a layer."""

    def __init__(self, M, K, N, block, gen, signs=None, out=torch.bfloat16):
        w = _weights(N, K, gen)
        self.N = N
        self.codes, self.scales = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
        if signs is None:
            bro.pack_weights(w, block, self.codes, self.scales)
        else:
            bro.pack_weights_rs(w, block, signs, self.codes, self.scales)
        ld = -(-N // 8) * 8                     # rows of the output start on 16 bytes
        self.y = torch.zeros(M, ld, dtype=out, device="cuda")[:, :N]
        self.ws = bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, M, block = case["kind"], case["M"], case["block"]
    s = {"case": case}
    if kind == "stack":
        d, kv, f = case["d"], case["kv"], case["f"]
        s["x_qkv"], s["x_o"], s["x_gu"] = (_activations(M, d, gen) for _ in range(3))
        s["qkv"], s["o"] = _Layer(M, d, d + 2 * kv, block, gen), _Layer(M, d, d, block, gen)
        s["gu"], s["down"] = _Layer(M, d, 2 * f, block, gen), _Layer(M, f, d, block, gen)
        return s
    K = case["K"]
    if kind == "linear":
        s["x"] = _activations(M, K, gen)
        s["signs"] = _signs(K, gen) if case["signs"] else None
        f32 = case["out"] == "f32"
        s["layer"] = _Layer(M, K, case["N"], block, gen, s["signs"], torch.float32 if f32 else torch.bfloat16)
        if f32:
            s["acodes"], s["ascales"] = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
    elif kind == "mlp":
        s["gate"], s["up"] = _activations(M, K, gen), _activations(M, K, gen)
        s["layer"] = _Layer(M, K, case["N"], block, gen)
    elif kind == "quantize":
        s["x"] = _weights(M, K, gen) if case["weights"] else _activations(M, K, gen)
        s["signs"] = _signs(K, gen) if case["signs"] else None
        s["layout"] = bro.LAYOUT_GEMM if case["layout"] == "gemm" else bro.LAYOUT_CANONICAL
        s["codes"], s["scales"] = bro.alloc_codes(M, K), bro.alloc_scales(M, K, s["layout"])
    elif kind == "formats":
        s["x"] = _activations(M, K, gen)
        s["deq"] = {f: torch.empty(M, K, dtype=torch.float32, device="cuda") for f in STUDY_FORMATS}
        s["ws"] = torch.empty(max(bro.fake_quantize_workspace_bytes(M, f) for f in STUDY_FORMATS), dtype=torch.uint8, device="cuda")
    else:
        s["x"] = _activations(M, K, gen)
        u8 = lambda: torch.empty(M, K // 32, dtype=torch.uint8, device="cuda")  # noqa: E731
        s["mask"], s["before"], s["after"] = u8(), u8(), u8()
        s["mse"] = torch.empty(M, K // 32, dtype=torch.float32, device="cuda")
        s["info"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        s["counts"] = torch.zeros(2, 3, dtype=torch.int64, device="cuda")
        s["hist"] = torch.zeros(2, 256, dtype=torch.int64, device="cuda")
        s["ws"] = torch.empty(bro.outlier_workspace_bytes(), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind, block = case["kind"], case["block"]
    if kind == "linear":
        L = s["layer"]
        if case["out"] == "f32":
            bro.rotate_quantize_mxfp4(s["x"], block, s["acodes"], s["ascales"], signs=s["signs"])
            bro.gemm_mxfp4(s["acodes"], s["ascales"], L.codes, L.scales, case["M"], L.N, case["K"], L.y)
        elif s["signs"] is not None:
            bro.linear_rs(s["x"], block, s["signs"], L.codes, L.scales, L.N, L.y, L.ws)
        else:
            bro.linear(s["x"], block, L.codes, L.scales, L.N, L.y, L.ws)
        return L.y
    if kind == "mlp":
        L = s["layer"]
        bro.swiglu_linear(s["gate"], s["up"], block, L.codes, L.scales, L.N, L.y, L.ws)
        return L.y
    if kind == "stack":
        qkv, o, gu, down, f = s["qkv"], s["o"], s["gu"], s["down"], case["f"]
        bro.linear(s["x_qkv"], block, qkv.codes, qkv.scales, qkv.N, qkv.y, qkv.ws)
        bro.linear(s["x_o"], block, o.codes, o.scales, o.N, o.y, o.ws)
        bro.linear(s["x_gu"], block, gu.codes, gu.scales, gu.N, gu.y, gu.ws)
        bro.swiglu_linear(gu.y[:, :f], gu.y[:, f:], block, down.codes, down.scales, down.N, down.y, down.ws)
        return [qkv.y, o.y, gu.y, down.y]
    if kind == "quantize":
        if case["weights"] and s["signs"] is None:
            bro.pack_weights(s["x"], block, s["codes"], s["scales"])
        elif case["weights"]:
            bro.pack_weights_rs(s["x"], block, s["signs"], s["codes"], s["scales"])
        else:
            bro.rotate_quantize_mxfp4(s["x"], block, s["codes"], s["scales"], s["layout"], signs=s["signs"])
        return [s["codes"], s["scales"]]
    if kind == "formats":
        for fmt, deq in s["deq"].items():
            bro.rotate_fake_quantize(s["x"], block, deq, fmt, workspace=s["ws"])
        return s["deq"]
    bro.outlier_groups(s["x"], s["mask"], s["info"], s["ws"])
    bro.group_scale_bytes(s["x"], 1, s["before"])
    bro.group_scale_bytes(s["x"], block, s["after"])
    bro.scale_inflation(s["before"], s["after"], s["mask"], s["counts"])
    bro.scale_histogram(s["after"], s["mask"], s["hist"])
    bro.group_quant_error(s["x"], block, s["mse"])
    return [s[k] for k in ("mask", "info", "before", "after", "counts", "hist", "mse")]


# ---- what a pass cannot do without -----------------------------------------------------------------------
def _layer_work(M, K, N, x_bytes=2, y_bytes=2):
    """x in, packed weights in (4-bit codes and one scale byte per 32), y out."""
    return x_bytes * M * K + 17 * N * K / 32 + y_bytes * M * N, 2.0 * M * K * N


def work(case):
    kind, M = case["kind"], case["M"]
    if kind == "stack":
        d, kv, f = case["d"], case["kv"], case["f"]
        parts = [_layer_work(M, d, d + 2 * kv), _layer_work(M, d, d), _layer_work(M, d, 2 * f), _layer_work(M, f, d, x_bytes=4)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    K = case["K"]
    e = M * K
    if kind in ("linear", "mlp"):
        y_bytes = 4 if case.get("out") == "f32" else 2
        b, f = _layer_work(M, K, case["N"], 4 if kind == "mlp" else 2, y_bytes)
        return {"bytes": b, "flops": f}
    stages = math.log2(case["block"] or K)
    if kind == "quantize":
        return {"bytes": e * (2 + 17 / 32), "flops": e * stages}
    if kind == "formats":                       # every call reads x and writes fp32
        return {"bytes": 6.0 * e * len(STUDY_FORMATS), "flops": e * stages * len(STUDY_FORMATS)}
    # four calls read x (outliers, bytes before, bytes after, error); one byte a group three times, one float
    return {"bytes": e * (4 * 2 + (3 + 4) / 32), "flops": 2 * e * stages}


def tolerance(case):
    kind = case["kind"]
    if kind in ("quantize", "formats"):
        return "exact"
    if kind == "scales":
        # fp32 sums of 32 squares in another order (against float64: rel 8e-8, max 4e-7); bytes and counts exact
        return {"rel": 3e-7, "max": 1.5e-6}
    # The codes are small multiples of powers of two, so nearly every fp32 sum is exact in any order (against
    # float64 the outputs showed no difference at all); a few last-bit roundings are left room for.
    if case.get("out") == "f32":
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 1e-4, "max": 1e-2}


# ---- the same outputs in 64 bits -------------------------------------------------------------------------
def _rotate64(x, block, signs=None):
    """x R in float64: the Walsh-Hadamard butterfly inside every block (0: the whole row), over sqrt(block)."""
    y = x.double() if signs is None else x.double() * signs.double()
    rows, K = y.shape
    B = block or K
    h = 1
    while h < B:
        y = y.view(rows, K // (2 * h), 2, h)
        y = torch.stack((y[:, :, 0] + y[:, :, 1], y[:, :, 0] - y[:, :, 1]), dim=2).view(rows, K)
        h *= 2
    return y / math.sqrt(B)


def _to_grid(a, grid):
    """Magnitudes to the nearest value of the E2M1 grid or of the integers 0..7 (halves to the even code)."""
    if grid == "int":
        return torch.round(a).clamp(max=7)
    step = torch.exp2(torch.floor(torch.log2(a.clamp(1, 6)))) / 2
    return (torch.round(a / step) * step).clamp(max=6)


def _quantised64(y, fmt):
    """Rotated values -> the values that the 4-bit format stands for, in float64."""
    rows, K = y.shape
    if fmt == "int4_row_asym":
        lo, hi = y.amin(1, True).clamp(max=0), y.amax(1, True).clamp(min=0)
        s = ((hi - lo) / 15).half().double()
        z = torch.round(-lo / s).clamp(max=15)
        return torch.where(s > 0, ((torch.round(y / s) + z).clamp(0, 15) - z) * s, torch.zeros_like(y))
    g = y.view(rows, K // 32, 32)
    amax = g.abs().amax(2, True)
    grid = "int" if fmt in ("mxint4", "bint4") else "e2m1"
    if fmt in ("mxfp4", "mxint4"):
        s = torch.exp2((torch.frexp(amax)[1] - 1).double() - 2)
    else:
        s = (amax / (7 if grid == "int" else 6)).half().double()
    q = torch.where(s > 0, _to_grid(g.abs() / s.clamp(min=2.0 ** -140), grid), torch.zeros_like(g))
    return (torch.sign(g) * q * s).view(rows, K)


def _linear64(x, w, block, signs=None):
    return _quantised64(_rotate64(x, block, signs), "mxfp4") @ _quantised64(_rotate64(w, block, signs), "mxfp4").T


def _gated64(gate, up):
    return (gate.double() * torch.sigmoid(gate.double()) * up.double()).to(torch.bfloat16)


def exact(case, seed):
    """What run returns, in float64; None for bytes, codes and counts, which are compared bit for bit."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, M, block = case["kind"], case["M"], case["block"]
    if kind == "quantize":
        return None
    if kind == "stack":
        d, kv, f = case["d"], case["kv"], case["f"]
        x_qkv, x_o, x_gu = (_activations(M, d, gen) for _ in range(3))
        qkv = _linear64(x_qkv, _weights(d + 2 * kv, d, gen), block)
        o = _linear64(x_o, _weights(d, d, gen), block)
        gu = _linear64(x_gu, _weights(2 * f, d, gen), block)
        h = _gated64(gu[:, :f].to(torch.bfloat16), gu[:, f:].to(torch.bfloat16))
        return [qkv, o, gu, _linear64(h, _weights(d, f, gen), block)]
    K = case["K"]
    x = _activations(M, K, gen)
    if kind == "linear":
        signs = _signs(K, gen) if case["signs"] else None
        return _linear64(x, _weights(case["N"], K, gen), block, signs)
    if kind == "mlp":
        h = _gated64(x, _activations(M, K, gen))
        return _linear64(h, _weights(case["N"], K, gen), block)
    y = _rotate64(x, block)
    if kind == "formats":
        return {fmt: _quantised64(y, fmt) for fmt in STUDY_FORMATS}
    mse = (y - _quantised64(y, "mxfp4")).square().view(M, K // 32, 32).mean(2)
    return [None, None, None, None, None, None, mse]
