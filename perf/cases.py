"""The work that users of libkmq have it do, as measurable cases: one pass each through the public entry points of
paper_2602_15563_b200.kmq on inputs of the shapes, bit widths and value distributions of the layers it is made for.

A case is a dict of plain values; "op" names the entry point (or the sequence of calls) that one pass goes through:

  linear          kmq_linear with weights packed once, as a serving program keeps them
  decode          every linear of a decoder stack for one token step, captured once as a CUDA graph and replayed
  host            kmq_linear_host: activations and result in pinned host memory
  dequant         kmq_dequant_to_bf16 of a whole matrix
  block_linear    the block format (shared codebook, bf16 scale per 64 inputs) in the interchange byte layout
  block_table     the block format in its own decode layout
  quantize_rows   float32 weights -> per-row codebooks and packed indices
  quantize_block  float32 weights -> block scales, shared codebook and packed indices
"""
import math
from functools import lru_cache
from statistics import NormalDist

import numpy as np
import torch

from paper_2602_15563_b200 import kmq

# upper ends of the ranges that drawn cases are taken from (each is reached by a listed case)
MAX_WEIGHTS = 8192 * 28672                # weights of one matrix
MAX_MACS = 16384 * 3072 * 1024            # multiply-adds of one call
MAX_STACK_BYTES = 24 * (9216 * 3072 + 3072 * 3072 + 16384 * 3072 + 3072 * 8192) * 2 // 8
MAX_QUANTIZED = 4096 * 4096               # weights quantised in one pass
ITERS = 20                                # Lloyd iterations of a fit
SAMPLES = 32768                           # values a shared codebook is fitted on


def listed():
    return [
        # the smallest layer of the benchmark configurations: nothing but the cost of a call
        {"name": "linear_tiny_b1_m1", "op": "linear", "N": 256, "K": 256, "bits": 1, "M": 1, "layout": "preferred"},
        # the layer the headline metric is quoted on, one token at a time
        {"name": "linear_4096_b2_m1", "op": "linear", "N": 4096, "K": 4096, "bits": 2, "M": 1, "layout": "preferred"},
        # the largest layer of the configurations (a down projection) under a small serving batch
        {"name": "linear_8192x28672_b4_m16", "op": "linear", "N": 8192, "K": 28672, "bits": 4, "M": 16,
         "layout": "preferred"},
        # prefill: a prompt of 1024 tokens through a stacked gate and up projection
        {"name": "linear_prefill_b2_m1024", "op": "linear", "N": 16384, "K": 3072, "bits": 2, "M": 1024,
         "layout": "preferred"},
        # weights left in the interchange layout (the binding's default), a row length that is only a multiple of 64
        # and a number of rows that is no multiple of anything
        {"name": "linear_ragged_canonical", "op": "linear", "N": 2999, "K": 2880, "bits": 1, "M": 3,
         "layout": "canonical"},
        # one token step of the ~3B-parameter decoder set of the configurations at batch 1
        {"name": "decode_3072x24_b2_m1", "op": "decode", "d": 3072, "hidden": 8192, "layers": 24, "bits": 2, "M": 1},
        # a caller whose activations live on the host
        {"name": "host_4096_b1_m1", "op": "host", "N": 4096, "K": 4096, "bits": 1, "M": 1, "layout": "preferred"},
        # weights materialised ahead of a standard matrix product
        {"name": "dequant_8192x28672_b4", "op": "dequant", "N": 8192, "K": 28672, "bits": 4, "layout": "preferred"},
        # the 1.25-bit micro-benchmark of the block format
        {"name": "block_table_8192_b1_m1", "op": "block_table", "N": 8192, "K": 8192, "bits": 1, "M": 1},
        # the block format in its byte layout under a small batch
        {"name": "block_linear_4096_b4_m8", "op": "block_linear", "N": 4096, "K": 4096, "bits": 4, "M": 8,
         "scale_order": "deferred"},
        # quantising a layer, per-row codebooks and block format
        {"name": "quantize_rows_4096_b4", "op": "quantize_rows", "N": 4096, "K": 4096, "bits": 4, "dist": "normal",
         "layout": "preferred"},
        {"name": "quantize_block_4096_b4", "op": "quantize_block", "N": 4096, "K": 4096, "bits": 4, "dist": "normal",
         "lambda": "absmax"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng):
    n = _log_int(rng, 256, 16384)
    return max(128, n // 128 * 128) if rng.random() < 0.6 else n      # layer widths are mostly multiples of 128


def _cols(rng, unit, hi=28672):
    """A row length: mostly a multiple of 128, sometimes of 64, sometimes only what the packing needs."""
    k, r = _log_int(rng, 256, hi), rng.random()
    step = 128 if r < 0.6 else 64 if r < 0.85 else unit
    step = math.lcm(step, unit)
    return max(step, k // step * step)


def draw(rng):
    op = rng.choice(["linear"] * 5 + ["decode", "host", "dequant", "block_table", "block_linear", "quantize_rows",
                                      "quantize_block"])
    bits = rng.choice([1, 2, 4])
    if op == "decode":
        d = 256 * rng.randint(4, 16)
        hidden = -(-d * 8 // 3) // 256 * 256
        m = 1 if rng.random() < 0.5 else rng.randint(2, 8)
        per_layer = sum(n * k for n, k in _stack_shapes(d, hidden)) * bits // 8
        layers = max(1, min(rng.randint(8, 48), MAX_STACK_BYTES // per_layer))
        return {"op": op, "d": d, "hidden": hidden, "layers": layers, "bits": bits, "M": m}
    if op.startswith("quantize"):
        n, k = _rows(rng), _cols(rng, 64 if op == "quantize_block" else 32)
        n = max(16, min(n, MAX_QUANTIZED // k))
        c = {"op": op, "N": n, "K": k, "bits": bits, "dist": rng.choice(["normal", "student_t", "laplace"])}
        if op == "quantize_rows":
            c["layout"] = rng.choice(["preferred", "canonical"])
        else:
            c["lambda"] = rng.choice(["absmax", "absmean"])
        return c
    block = op.startswith("block")
    n, k = _rows(rng), _cols(rng, 64 if block else 32 // bits)
    n = max(16, min(n, MAX_WEIGHTS // k))
    if op == "dequant":
        return {"op": op, "N": n, "K": k, "bits": bits, "layout": rng.choice(["preferred", "canonical"])}
    if op == "block_table":
        return {"op": op, "N": n, "K": k, "bits": bits, "M": rng.choice([1, 1, 2, 4])}
    if op == "block_linear":
        bits = rng.choice([1, 2, 4, 8])
        return {"op": op, "N": n, "K": k, "bits": bits, "M": _log_int(rng, 1, 16),
                "scale_order": rng.choice(["deferred", "deferred", "direct"])}
    layout = "canonical" if rng.random() < 0.2 else "preferred"
    r = rng.random()
    m = 1 if r < 0.4 else _log_int(rng, 2, 64)
    if op == "linear" and layout == "preferred" and r > 0.8:
        m = _log_int(rng, 65, 1024)                                   # prefill
    m = max(1, min(m, MAX_MACS // (n * k)))
    return {"op": op, "N": n, "K": k, "bits": bits, "M": m, "layout": layout}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
@lru_cache(maxsize=None)
def _levels(bits):
    """The 2^bits centroids of 1-D k-means on a standard normal (Lloyd on its quantiles), ascending."""
    q, n = 1 << bits, 1 << 14
    inv = NormalDist().inv_cdf
    v = np.array([inv((i + 0.5) / n) for i in range(n)])
    c = np.array([inv((i + 0.5) / q) for i in range(q)])
    for _ in range(60):
        edges = np.concatenate([[0], np.searchsorted(v, 0.5 * (c[1:] + c[:-1])), [n]])
        c = np.array([v[a:b].mean() if b > a else m for a, b, m in zip(edges[:-1], edges[1:], c)])
    return c


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _indices(g, N, K, bits):
    """uint8 [N, K]: nearest-centroid indices of normally distributed weights."""
    c = _levels(bits)
    mids = torch.tensor(0.5 * (c[1:] + c[:-1]), dtype=torch.float32, device="cuda")
    idx = torch.empty((N, K), dtype=torch.uint8, device="cuda")
    rows = max(1, (1 << 26) // K)
    for r in range(0, N, rows):
        w = torch.randn((min(rows, N - r), K), device="cuda", generator=g)
        idx[r:r + rows] = torch.bucketize(w, mids, out_int32=True)
    return idx


def _codebooks(g, N, bits):
    """bf16 [N, 2^bits], ascending: the k-means centroids of rows whose weights have a std near 0.02."""
    std = 0.02 * (1.0 + 0.1 * torch.randn((N, 1), device="cuda", generator=g).clamp(-3, 3))
    c = torch.tensor(_levels(bits), dtype=torch.float32, device="cuda")
    return (c * std).to(torch.bfloat16)


def _activations(g, M, K):
    return torch.randn((M, K), device="cuda", generator=g).to(torch.bfloat16)


def _weights(g, N, K, dist):
    """float32 [N, K] weights of standard deviation close to 0.02."""
    if dist == "normal":
        return torch.randn((N, K), device="cuda", generator=g) * 0.02
    if dist == "laplace":
        u = torch.rand((N, K), device="cuda", generator=g) - 0.5
        return -0.014 * u.sign() * torch.log1p(-2 * u.abs().clamp(max=0.4999999))
    chi2 = sum(torch.randn((N, K), device="cuda", generator=g).square_() for _ in range(5))
    t = torch.randn((N, K), device="cuda", generator=g) / (chi2 / 5).sqrt_()
    return t * (0.02 / math.sqrt(5.0 / 3.0))


def _layout(case, bits, M):
    if case.get("layout") == "canonical":
        return kmq.KMQ_LAYOUT_CANONICAL
    return kmq.kmq_preferred_layout(case["N"], case["K"], bits, M)


def _packed(g, N, K, bits, layout):
    out = torch.empty(kmq.kmq_packed_bytes(N, K, bits, layout) // 4, dtype=torch.int32, device="cuda")
    kmq.kmq_pack(_indices(g, N, K, bits), N, K, bits, out, layout=layout)
    return out


def _workspace(nbytes):
    return torch.empty(max(nbytes, 16), dtype=torch.uint8, device="cuda")


def _stack_shapes(d, hidden):
    """(N, K) of the linears of one decoder layer: fused QKV, attention output, stacked gate and up, down."""
    return [(3 * d, d), (d, d), (2 * hidden, d), (d, hidden)]


def _prepare_stack(case, g):
    bits, M, L = case["bits"], case["M"], case["layers"]
    shapes = _stack_shapes(case["d"], case["hidden"])
    calls, ys, ws_bytes = [], [torch.zeros((L, M, n), dtype=torch.bfloat16, device="cuda") for n, _ in shapes], 16
    for layer in range(L):
        for j, (N, K) in enumerate(shapes):
            layout = kmq.kmq_preferred_layout(N, K, bits, M)
            ws_bytes = max(ws_bytes, kmq.kmq_workspace_bytes(N, K, bits, M, layout))
            calls.append((_packed(g, N, K, bits, layout), _codebooks(g, N, bits), _activations(g, M, K), ys[j][layer],
                          N, K, layout))
    ws = _workspace(ws_bytes)

    def step(todo):
        for packed, cb, x, y, N, K, layout in todo:
            kmq.kmq_linear(packed, cb, x, y, N, K, bits, M, ws, ws_bytes, layout=layout)

    step(calls[:len(shapes)])                       # every kernel once before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(calls)
    return {"graph": graph, "calls": calls, "ws": ws, "y": ys}


def prepare(case, seed):
    g, op = _gen(seed), case["op"]
    s = {"case": dict(case)}
    if op == "decode":
        s.update(_prepare_stack(case, g))
        return s
    N, K, bits = case["N"], case["K"], case["bits"]
    if op in ("linear", "host"):
        M = case["M"]
        s["layout"] = _layout(case, bits, M)
        s["packed"], s["cb"] = _packed(g, N, K, bits, s["layout"]), _codebooks(g, N, bits)
        s["x"], s["y"] = _activations(g, M, K), torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
        s["ws_bytes"] = kmq.kmq_workspace_bytes(N, K, bits, M, s["layout"])
        s["ws"] = _workspace(s["ws_bytes"])
        if op == "host":
            s["x_host"] = s["x"].cpu().pin_memory()
            s["y_host"] = torch.zeros((M, N), dtype=torch.bfloat16).pin_memory()
    elif op == "dequant":
        s["layout"] = _layout(case, bits, 1)
        s["packed"], s["cb"] = _packed(g, N, K, bits, s["layout"]), _codebooks(g, N, bits)
        s["W"] = torch.empty((N, K), dtype=torch.bfloat16, device="cuda")
    elif op in ("block_linear", "block_table"):
        M = case["M"]
        wq = torch.empty(kmq.kmq_block_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
        kmq.kmq_block_pack(_indices(g, N, K, bits), N, K, bits, wq)
        # largest magnitude of 64 normal weights of std 0.02, and a codebook inside [-1, 1]
        scales = 0.048 + 0.008 * torch.randn((N, K // 64), device="cuda", generator=g)
        scales = scales.clamp(0.02, 0.1).to(torch.bfloat16)
        s["cb"] = torch.tensor(_levels(bits) / 2.4, device="cuda").clamp(-1, 1).to(torch.bfloat16)
        s["x"], s["y"] = _activations(g, M, K), torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
        if op == "block_linear":
            s["wq"], s["scales"] = wq, scales
            s["order"] = kmq.KMQ_SCALE_DIRECT if case["scale_order"] == "direct" else kmq.KMQ_SCALE_DEFERRED
        else:
            s["table"] = torch.empty(kmq.kmq_block_table_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
            kmq.kmq_block_table_pack(wq, scales, N, K, bits, s["table"])
            s["ws_bytes"] = kmq.kmq_block_table_workspace_bytes(N, K, bits)
            s["ws"] = _workspace(s["ws_bytes"])
    elif op == "quantize_rows":
        s["layout"] = _layout(case, bits, 1)
        s["W"] = _weights(g, N, K, case["dist"])
        s["cb"] = torch.empty((N, 1 << bits), dtype=torch.bfloat16, device="cuda")
        s["packed"] = torch.empty(kmq.kmq_packed_bytes(N, K, bits, s["layout"]) // 4, dtype=torch.int32, device="cuda")
    else:
        s["W"] = _weights(g, N, K, case["dist"])
        s["lam"] = kmq.KMQ_LAMBDA_ABSMAX if case["lambda"] == "absmax" else kmq.KMQ_LAMBDA_ABSMEAN
        s["scales"] = torch.empty((N, K // 64), dtype=torch.bfloat16, device="cuda")
        s["cb"] = torch.empty(1 << bits, dtype=torch.bfloat16, device="cuda")
        s["wq"] = torch.empty(kmq.kmq_block_packed_bytes(N, K, bits), dtype=torch.uint8, device="cuda")
        s["sample"] = torch.empty(SAMPLES, dtype=torch.float32, device="cuda")
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(s):
    c = s["case"]
    op = c["op"]
    if op == "decode":
        s["graph"].replay()
        return s["y"]
    N, K, bits = c["N"], c["K"], c["bits"]
    if op == "linear":
        kmq.kmq_linear(s["packed"], s["cb"], s["x"], s["y"], N, K, bits, c["M"], s["ws"], s["ws_bytes"],
                       layout=s["layout"])
        return s["y"]
    if op == "host":
        kmq.kmq_linear_host(s["packed"], s["cb"], s["x_host"].data_ptr(), s["y_host"].data_ptr(), N, K, bits, c["M"],
                            s["x"], s["y"], s["ws"], s["ws_bytes"], layout=s["layout"])
        return s["y_host"]
    if op == "dequant":
        kmq.kmq_dequant_to_bf16(s["packed"], s["cb"], s["W"], N, K, bits, layout=s["layout"])
        return s["W"]
    if op == "block_linear":
        kmq.kmq_block_linear(s["wq"], s["scales"], s["cb"], s["x"], s["y"], N, K, bits, c["M"], scale_order=s["order"])
        return s["y"]
    if op == "block_table":
        kmq.kmq_block_table_linear(s["table"], s["cb"], s["x"], s["y"], N, K, bits, c["M"], s["ws"], s["ws_bytes"])
        return s["y"]
    if op == "quantize_rows":
        kmq.kmq_quantize_rows(s["W"], N, K, bits, ITERS, s["layout"], s["cb"], s["packed"])
        return {"codebooks": s["cb"], "packed": s["packed"]}
    kmq.kmq_block_quantize(s["W"], N, K, bits, s["lam"], ITERS, SAMPLES, s["scales"], s["cb"], s["wq"], s["sample"])
    return {"scales": s["scales"], "codebook": s["cb"], "wq": s["wq"]}


# --------------------------------------------------------------------------
# what a pass cannot do without, and how close two correct results are
# --------------------------------------------------------------------------
def _linear_work(N, K, bits, M):
    return {"bytes": N * K * bits / 8 + N * (1 << bits) * 2 + M * (K + N) * 2, "flops": 2.0 * M * N * K}


def work(case):
    op, bits = case["op"], case["bits"]
    if op == "decode":
        per = [_linear_work(n, k, bits, case["M"]) for n, k in _stack_shapes(case["d"], case["hidden"])]
        return {key: case["layers"] * sum(w[key] for w in per) for key in ("bytes", "flops")}
    N, K = case["N"], case["K"]
    if op in ("linear", "host"):
        return _linear_work(N, K, bits, case["M"])
    if op == "dequant":
        return {"bytes": N * K * bits / 8 + N * (1 << bits) * 2 + 2.0 * N * K, "flops": 0}
    if op in ("block_linear", "block_table"):
        M = case["M"]
        return {"bytes": N * K * (bits + 0.25) / 8 + (1 << bits) * 2 + M * (K + N) * 2, "flops": 2.0 * M * N * K}
    if op == "quantize_rows":
        return {"bytes": 4.0 * N * K + N * K * bits / 8 + N * (1 << bits) * 2, "flops": 0}
    return {"bytes": 4.0 * N * K + N * K * (bits + 0.25) / 8 + (1 << bits) * 2, "flops": 0}


def tolerance(case):
    """Copies of stored centroids, indices, scales and codebooks are exact.  A layer's output is an fp32 sum rounded to
    bf16: another order of the sum moves some values by one bf16 step (at most 2^-7 of the value)."""
    if case["op"] == "dequant" or case["op"].startswith("quantize"):
        return "exact"
    return {"rel": 4e-3, "max": 0.02}
