"""Performance cases of the FP8 library: what its users have it do.

Every case goes through the package's public entry points, as a program that
uses them would call them, over the sizes of the repository's own workloads
(workloads.py, the benchmark and the tests) and odd sizes between them.  A
case is a dict of plain values; its "kind" names the path:

  tensor   fp32 A and B -> per-tensor scales and codes -> dense GEMM, eager:
           the library's smallest whole computation, and its ragged forms
  decode   one decode step's four projections (per-row activation
           quantisation + skinny GEMM each), captured once in a CUDA graph
           and replayed, as a serving loop runs it
  dense    one eager dense GEMM on resident codes
  layer    a prefill layer: four per-row activation quantisations and the
           four GEMMs as one grouped launch (GroupedGraph)
  sparse   one eager 2:4 GEMM with sparse weights and transposed output
  mx       block-scaled linear: quantise the activations, then the GEMM
  prune    weights to 2:4 and back: per-row quantise, compress, decompress
           (the dense comparison form)
  load24   weights to 2:4 in one pass (fused quantise + compress)
  serve    a burst of requests of uneven sizes through the request server
"""
from __future__ import annotations

import math
import random

import torch

import paper_2602_10262_gb300 as gb
from paper_2602_10262_gb300.server import Server

FMAX = {gb.E4M3: 448.0, gb.E5M2: 57344.0}
FDTYPE = {gb.E4M3: torch.float8_e4m3fn, gb.E5M2: torch.float8_e5m2}

# (N, K) and 2:4 flag of the weights that a serving case keeps resident
SERVE_WEIGHTS = ((14336, 4096, False), (4096, 14336, False), (8192, 8192, True), (4096, 4096, True))


def listed():
    return [
        # The smallest whole computation: 256^3, per-tensor scales, fp32 out,
        # where launches and latency count (the single-call configuration).
        {"name": "tensor_256", "kind": "tensor", "M": 256, "N": 256, "K": 256, "b_format": 0, "out": 0},
        # Ragged sizes as real tables have them: odd N (unaligned output
        # rows), K that is no multiple of a tile, E4M3 x E5M2, bf16 out.
        {"name": "tensor_ragged", "kind": "tensor", "M": 1000, "N": 3001, "K": 4100, "b_format": 1, "out": 1},
        # One decode step of a 4096-wide layer for 16 sequences.
        {"name": "decode_16", "kind": "decode", "tokens": 16, "d": 4096, "qkv": 12288, "ffn": 14336},
        # A chunk of a prompt through one projection: a mid-size product.
        {"name": "dense_chunk_512", "kind": "dense", "M": 512, "N": 12288, "K": 4096, "b_format": 0, "out": 1},
        # Square product of the shape sweep, bound by the tensor cores.
        {"name": "dense_8192", "kind": "dense", "M": 8192, "N": 8192, "K": 8192, "b_format": 0, "out": 1},
        # The transformer layer of 8 x 2048 tokens: the largest case.
        {"name": "layer_16384", "kind": "layer", "tokens": 16384, "d": 4096, "qkv": 12288, "ffn": 14336},
        # 2:4 weights under a small batch: a skinny sparse product.
        {"name": "sparse_decode_128", "kind": "sparse", "tokens": 128, "N": 8192, "K": 8192, "out": 1},
        # 2:4 weights under a prompt: a large sparse product.
        {"name": "sparse_prefill_4096", "kind": "sparse", "tokens": 4096, "N": 14336, "K": 4096, "out": 1},
        # Block-scaled linear layer of a prompt: quantise + GEMM.
        {"name": "mx_4096", "kind": "mx", "M": 4096, "N": 14336, "K": 4096, "out": 1},
        # E5M2 weights pruned to 2:4, and expanded again for the dense
        # comparison (encode and decode of the compressed form).
        {"name": "prune_8192", "kind": "prune", "R": 8192, "C": 8192, "format": 1},
        # An up-projection's weights loaded as 2:4 in one pass.
        {"name": "load24_14336", "kind": "load24", "R": 14336, "C": 4096},
        # A burst at the request server: two tenants, small requests beside
        # large ones, dense and 2:4 weights.
        {"name": "serve_32", "kind": "serve", "requests": 32, "m_max": 1024, "mix": 2},
    ]


def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, int(round(v / step)) * step)


def draw(rng: random.Random):
    kind = rng.choice(("tensor", "tensor", "decode", "dense", "dense", "layer", "sparse", "sparse", "mx", "mx",
                       "prune", "load24", "serve"))
    if kind == "tensor":
        return {"kind": kind, "M": _log(rng, 1, 8192), "N": _log(rng, 16, 8192), "K": _log(rng, 16, 8192, 4),
                "b_format": rng.randint(0, 1), "out": rng.randint(0, 1)}
    if kind == "decode":
        d = _log(rng, 1024, 8192, 16)
        return {"kind": kind, "tokens": _log(rng, 1, 128), "d": d, "qkv": 3 * d, "ffn": _log(rng, 2 * d, 4 * d, 16)}
    if kind == "dense":
        return {"kind": kind, "M": _log(rng, 1, 16384), "N": _log(rng, 64, 14336), "K": _log(rng, 64, 14336),
                "b_format": rng.randint(0, 1), "out": rng.randint(0, 1)}
    if kind == "layer":
        d = _log(rng, 1024, 4096, 16)
        return {"kind": kind, "tokens": _log(rng, 256, 16384), "d": d, "qkv": 3 * d,
                "ffn": min(14336, _log(rng, 2 * d, 4 * d, 16))}
    if kind == "sparse":
        return {"kind": kind, "tokens": _log(rng, 1, 8192), "N": _log(rng, 256, 14336), "K": _log(rng, 256, 14336, 128),
                "out": rng.randint(0, 1)}
    if kind == "mx":
        return {"kind": kind, "M": _log(rng, 1, 8192), "N": _log(rng, 64, 14336), "K": _log(rng, 64, 14336, 32),
                "out": rng.randint(0, 1)}
    if kind == "prune":
        return {"kind": kind, "R": _log(rng, 1, 16384), "C": _log(rng, 64, 14336, 4), "format": rng.randint(0, 1)}
    if kind == "load24":
        return {"kind": kind, "R": _log(rng, 1, 16384), "C": _log(rng, 128, 16384, 128)}
    return {"kind": "serve", "requests": rng.randint(4, 64), "m_max": _log(rng, 64, 4096), "mix": rng.randint(0, 999)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)


def _code_buffer(rows, cols):
    """Codes [rows, cols] whose rows start on 16-byte boundaries, as the GEMMs want them."""
    ld = (cols + 15) // 16 * 16
    return torch.empty((rows, ld), dtype=torch.uint8, device="cuda")[:, :cols]


def _quantize(x, fmt, mode=1):
    f = gb.fp8_quantize_e5m2 if fmt == gb.E5M2 else gb.fp8_quantize_e4m3
    return f(x, mode, q=_code_buffer(*x.shape))


def _projections(case):
    """(N, K) of the four projections of a layer."""
    d, qkv, ffn = case["d"], case["qkv"], case["ffn"]
    return ((qkv, d), (d, d), (ffn, d), (d, ffn))


def _serve_mix(case):
    """(tenant, weight index, M) of every request: the small tenant's M up to
    64, the other's from there to m_max, log-uniform."""
    rng = random.Random(case["mix"])
    mix = []
    for i in range(case["requests"]):
        tenant = i % 2
        lo, hi = (1, min(64, case["m_max"])) if tenant == 0 else (min(64, case["m_max"]), case["m_max"])
        mix.append((tenant, rng.randrange(len(SERVE_WEIGHTS)), _log(rng, lo, hi)))
    return mix


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    s = {"case": case}
    if kind == "tensor":
        s["x"], s["w"] = _randn(g, case["M"], case["K"]), _randn(g, case["N"], case["K"])
        s["A"], s["B"] = _code_buffer(case["M"], case["K"]), _code_buffer(case["N"], case["K"])
    elif kind == "decode":
        s["parts"] = []
        for n, k in _projections(case):
            x, w = _randn(g, case["tokens"], k), _randn(g, n, k)
            B, dB = _quantize(w, gb.E4M3)
            q, d = _code_buffer(case["tokens"], k), torch.empty(case["tokens"], device="cuda")
            C = torch.empty((case["tokens"], n), dtype=torch.bfloat16, device="cuda")
            s["parts"].append((x, q, d, B, dB, C))
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode(s["parts"])                        # warm-up before the capture
        torch.cuda.current_stream().wait_stream(side)
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _decode(s["parts"])
    elif kind == "dense":
        s["A"], s["dA"] = _quantize(_randn(g, case["M"], case["K"]), gb.E4M3)
        s["B"], s["dB"] = _quantize(_randn(g, case["N"], case["K"]), case["b_format"])
    elif kind == "layer":
        s["parts"], probs = [], []
        for n, k in _projections(case):
            x, w = _randn(g, case["tokens"], k), _randn(g, n, k)
            B, dB = _quantize(w, gb.E4M3)
            q, d = _code_buffer(case["tokens"], k), torch.empty(case["tokens"], device="cuda")
            C = torch.empty((case["tokens"], n), dtype=torch.bfloat16, device="cuda")
            s["parts"].append((x, q, d, B, dB, C))
            probs.append(gb.make_problem(q, B, d, 1, dB, 1, C))
        s["graph"] = gb.GroupedGraph(probs)
    elif kind == "sparse":
        s["x"], s["dx"] = _quantize(_randn(g, case["tokens"], case["K"]), gb.E4M3)
        _, s["dW"], s["vals"], s["meta"] = gb.fp8_quantize_e4m3_prune24(_randn(g, case["N"], case["K"]))
    elif kind == "mx":
        s["x"] = _randn(g, case["M"], case["K"])
        s["q"] = _code_buffer(case["M"], case["K"])
        w = _randn(g, case["N"], case["K"])
        s["B"], s["SB"] = gb.fp8_quantize_mx(w, q=_code_buffer(case["N"], case["K"]))
    elif kind in ("prune", "load24"):
        s["w"] = _randn(g, case["R"], case["C"])
    else:
        s["server"] = Server(num_tenants=2, latency_tenant=0, pool_bytes=1 << 30)
        handles = []
        for n, k, sparse in SERVE_WEIGHTS:
            w = _randn(g, n, k)
            if sparse:
                _, dW, vals, meta = gb.fp8_quantize_e4m3_prune24(w)
                handles.append(s["server"].register_weight(n, k, vals, dW, 1, meta))
            else:
                W, dW = _quantize(w, gb.E4M3)
                handles.append(s["server"].register_weight(n, k, W, dW, 1))
        s["requests"] = []
        for tenant, i, m in _serve_mix(case):
            n, k, _ = SERVE_WEIGHTS[i]
            out = torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
            s["requests"].append((tenant, handles[i], m, _randn(g, m, k), k, out, n))
        torch.cuda.synchronize()                       # the server works on streams of its own
    return s


# ------------------------------------------------------------------ one pass

def _decode(parts):
    for x, q, d, B, dB, C in parts:
        gb.fp8_quantize_e4m3(x, 1, q=q, dequant_scale=d)
        gb.gemm_fp8_dense(q, B, d, 1, dB, 1, C=C)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tensor":
        A, dA = gb.fp8_quantize_e4m3(state["x"], 0, q=state["A"])
        quantize = gb.fp8_quantize_e5m2 if case["b_format"] == gb.E5M2 else gb.fp8_quantize_e4m3
        B, dB = quantize(state["w"], 0, q=state["B"])
        C = gb.gemm_fp8_dense_fmt(A, B, dA, 0, dB, 0, 1.0, case["out"], gb.E4M3, case["b_format"])
        return [C, A, dA, B, dB]
    if kind == "decode":
        state["graph"].replay()
        return [p[5] for p in state["parts"]]
    if kind == "dense":
        return gb.gemm_fp8_dense_fmt(state["A"], state["B"], state["dA"], 1, state["dB"], 1, 1.0, case["out"],
                                     gb.E4M3, case["b_format"])
    if kind == "layer":
        for x, q, d, _, _, _ in state["parts"]:
            gb.fp8_quantize_e4m3(x, 1, q=q, dequant_scale=d)
        state["graph"].launch()
        return [p[5] for p in state["parts"]]
    if kind == "sparse":
        return gb.gemm_fp8_sparse24(state["vals"], state["meta"], state["x"], state["dW"], 1, state["dx"], 1,
                                    out_dtype=case["out"], out_transposed=True)
    if kind == "mx":
        A, SA = gb.fp8_quantize_mx(state["x"], q=state["q"])
        return gb.gemm_fp8_mx(A, SA, state["B"], state["SB"], out_dtype=case["out"])
    if kind == "prune":
        quantize = gb.fp8_quantize_e5m2 if case["format"] == gb.E5M2 else gb.fp8_quantize_e4m3
        W, dW = quantize(state["w"], 1)
        vals, meta = gb.prune24_compress(W)
        return [W, dW, vals, meta, gb.prune24_decompress(vals, meta, case["C"])]
    if kind == "load24":
        return list(gb.fp8_quantize_e4m3_prune24(state["w"]))
    server = state["server"]
    tickets = [server.submit(tenant, h, m, x, ldx, out, ldo)
               for tenant, h, m, x, ldx, out, ldo in state["requests"]]
    for t in tickets:
        r = server.wait(t)
        if r is None or r.status != 0:
            raise RuntimeError(f"request failed: {r}")
    return [r[5] for r in state["requests"]]


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind == "tensor":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 5 * (M + N) * K + (2 if case["out"] else 4) * M * N + 8, "flops": 2 * M * N * K}
    if kind in ("decode", "layer"):
        m = case["tokens"]
        return {"bytes": sum(4 * m * k + n * k + 4 * n + 2 * m * n for n, k in _projections(case)),
                "flops": sum(2 * m * n * k for n, k in _projections(case))}
    if kind == "dense":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": (M + N) * (K + 4) + (2 if case["out"] else 4) * M * N, "flops": 2 * M * N * K}
    if kind == "sparse":
        m, N, K = case["tokens"], case["N"], case["K"]
        return {"bytes": N * (K * 5 // 8 + 4) + m * (K + 4) + (2 if case["out"] else 4) * m * N,
                "flops": m * N * K}                    # two of four products
    if kind == "mx":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * M * K + N * (K + K // 32) + (2 if case["out"] else 4) * M * N, "flops": 2 * M * N * K}
    if kind == "prune":
        R, C = case["R"], case["C"]                    # W, kept codes, metadata, the expanded codes
        return {"bytes": R * (4 * C + C + C // 2 + (C + 7) // 8 + C + 4), "flops": R * C}
    if kind == "load24":
        R, C = case["R"], case["C"]
        return {"bytes": R * (4 * C + C + C // 2 + C // 8 + 4), "flops": R * C}
    mix = _serve_mix(case)
    used = {i for _, i, _ in mix}
    total = sum(n * (k * 5 // 8 if sp else k) + 4 * n for i, (n, k, sp) in enumerate(SERVE_WEIGHTS) if i in used)
    flops = 0
    for _, i, m in mix:
        n, k, sp = SERVE_WEIGHTS[i]
        total += 4 * m * k + 2 * m * n
        flops += m * n * k * (1 if sp else 2)
    return {"bytes": total, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits

def _codes64(x, fmt, per_row):
    """(decoded codes, dequantisation factors) in 64 bits of a scaled cast:
    s = fl32(T / amax), codes the format's round-to-nearest cast of
    fl32(x * s), factor amax / T (1 for an all-zero row)."""
    amax = x.abs().amax(dim=1, keepdim=True) if per_row else x.abs().amax().reshape(1, 1)
    t = torch.full_like(amax, FMAX[fmt])
    zero = amax == 0
    s = torch.where(zero, torch.ones_like(amax), torch.div(t, amax))
    q = (x * s).clamp(-FMAX[fmt], FMAX[fmt]).to(FDTYPE[fmt])
    d = torch.where(zero, torch.ones_like(amax).double(), torch.div(amax.double(), t.double()))
    return q, d


def _prune64(q):
    """The 2:4 form of codes [R, C]: of every four the two of largest
    magnitude (the earlier on a tie), the others zero."""
    R, C = q.shape
    key = (q.view(torch.uint8).to(torch.int32) & 127).reshape(R, C // 4, 4) * 4 + torch.arange(
        3, -1, -1, device=q.device, dtype=torch.int32)
    kept = torch.zeros_like(key, dtype=torch.bool).scatter_(2, key.topk(2, dim=2).indices, True)
    return q.to(torch.float64) * kept.reshape(R, C)


def _mx64(x):
    """Block-scaled values [R, C] in 64 bits: 32 columns share 2^e, e =
    floor(log2 amax) - 8; the codes are the saturating cast of x / 2^e."""
    R, C = x.shape
    b = x.reshape(R, C // 32, 32)
    amax = b.abs().amax(dim=2, keepdim=True)
    e = torch.frexp(amax).exponent.double() - 1 - 8
    e = torch.where(amax == 0, torch.full_like(e, -127.0), e.clamp(-127, 127))
    scale = torch.pow(torch.tensor(2.0, dtype=torch.float64, device=x.device), e)
    q = (b.double() / scale).float().clamp(-448, 448).to(torch.float8_e4m3fn).double()
    return (q * scale).reshape(R, C)


def _linear64(x, w, x_fmt=gb.E4M3, w_fmt=gb.E4M3, per_row=True, sparse=False):
    qx, dx = _codes64(x, x_fmt, per_row)
    qw, dw = _codes64(w, w_fmt, per_row)
    wv = _prune64(qw) if sparse else qw.double()
    return (qx.double() @ wv.T) * dx * dw.reshape(1, -1)


def exact(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "tensor":
        x, w = _randn(g, case["M"], case["K"]), _randn(g, case["N"], case["K"])
        dA, dB = _codes64(x, gb.E4M3, False)[1], _codes64(w, case["b_format"], False)[1]
        return [_linear64(x, w, w_fmt=case["b_format"], per_row=False), None, dA.reshape(1), None, dB.reshape(1)]
    if kind in ("decode", "layer"):
        out = []
        for n, k in _projections(case):
            x, w = _randn(g, case["tokens"], k), _randn(g, n, k)
            out.append(_linear64(x, w))
            del x, w
        return out
    if kind == "dense":
        x = _randn(g, case["M"], case["K"])
        return _linear64(x, _randn(g, case["N"], case["K"]), w_fmt=case["b_format"])
    if kind == "sparse":
        x = _randn(g, case["tokens"], case["K"])
        return _linear64(x, _randn(g, case["N"], case["K"]), sparse=True)
    if kind == "mx":
        x = _mx64(_randn(g, case["M"], case["K"]))
        return x @ _mx64(_randn(g, case["N"], case["K"])).T
    if kind == "prune":
        w = _randn(g, case["R"], case["C"])
        return [None, _codes64(w, case["format"], True)[1].reshape(-1), None, None, None]
    if kind == "load24":
        w = _randn(g, case["R"], case["C"])
        return [None, _codes64(w, gb.E4M3, True)[1].reshape(-1), None, None]
    weights = [_randn(g, n, k) for n, k, _ in SERVE_WEIGHTS]
    out = []
    for _, i, m in _serve_mix(case):
        n, k, sparse = SERVE_WEIGHTS[i]
        out.append(_linear64(_randn(g, m, k), weights[i], sparse=sparse))
    return out
