"""The GEMM calls that are timed: inputs, the call, its exact result and its work.

A case is one GEMM (``"kind": "gemm"``) or the four weight GEMMs of a
transformer layer (``"kind": "layer"``: QKV, attention output, MLP up, MLP
down; one call each), made through the binding of the C ABI the way a program
that uses the library does: operands, weights and output buffers are in device
memory, the stream is torch's current one.

Types (``dtype``): "int8" (exact int32 C), "int8_int16" and "int8_int8"
(requantised C, right shift ``shift``) and "bf16".  Layouts: "row" is B stored
K x N, "col" is B stored N x K.  Entries follow the repository's workloads:
int8 uniform on [-128, 127] (weights of a layer on [-64, 63]), bf16 N(0, 1)
times ``b_scale`` for B.
"""
import math

import torch

from paper_2512_13282_gb300 import gemm as G

_OUT = {"int8": torch.int32, "int8_int16": torch.int16, "int8_int8": torch.int8, "bf16": torch.bfloat16}


def _gemm(name, dtype, M, N, K, layout, b_scale=1.0, shift=0):
    return {"name": name, "kind": "gemm", "dtype": dtype, "M": M, "N": N, "K": K, "layout": layout,
            "b_scale": b_scale, "shift": shift}


def _layer(name, dtype, M, d, ffn, layout, shift=0):
    return {"name": name, "kind": "layer", "dtype": dtype, "M": M, "d": d, "ffn": ffn, "layout": layout,
            "b_scale": 0.02, "shift": shift}


def listed():
    return [
        # the smallest call: one tile's worth of int8 work, where the time is latency, launches and the host
        _gemm("int8_256", "int8", 256, 256, 256, "row"),
        # a small bf16 block of an operator-by-operator program (square sweep)
        _gemm("bf16_512", "bf16", 512, 512, 512, "col"),
        # a mid-sized int8 GEMM: a few tiles per SM, operands small enough to sit in L2 (square sweep)
        _gemm("int8_2048", "int8", 2048, 2048, 2048, "col"),
        # the ordinary compute-bound call of each type (square sweep)
        _gemm("bf16_4096", "bf16", 4096, 4096, 4096, "col"),
        _gemm("int8_4096", "int8", 4096, 4096, 4096, "col"),
        # the largest call of the benchmark, B row-major
        _gemm("int8_8192", "int8", 8192, 8192, 8192, "row"),
        # one token through a layer's weights, stored K x N: four matrix-vector products
        _layer("bf16_layer_1", "bf16", 1, 4096, 11008, "row"),
        # a small decode batch through int8 weights stored N x K
        _layer("int8_layer_16", "int8", 16, 4096, 11008, "col"),
        # a large decode batch (or a short prompt) through bf16 weights
        _layer("bf16_layer_128", "bf16", 128, 4096, 11008, "col"),
        # prefill of a quantised MLP: long K, int8 activations in and out
        _gemm("int8_int8_2048x4096x11008", "int8_int8", 2048, 4096, 11008, "col", shift=14),
        # sizes no tile divides, and a B row pitch (3000 bytes) that is not a multiple of 16 bytes
        _gemm("bf16_1000x1500x3000", "bf16", 1000, 1500, 3000, "row"),
        # a tall activation matrix against a narrow weight (a router or a low-rank factor), B row-major
        _gemm("int8_8192x64x8192", "int8", 8192, 64, 8192, "row"),
    ]


_DTYPES = ("int8", "bf16", "int8", "bf16", "int8_int16", "int8_int8")
_MAX_MACS = 8192 ** 3


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]: any integer, a multiple of 16, or one of 256."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    step = rng.choice((1, 16, 16, 256))
    return int(min(hi, max(lo, max(1, round(v / step)) * step)))


def _shift(dtype, K):
    """Keeps most requantised sums inside the output range: a sum has about 13 + log2(K) / 2 bits."""
    bits = {"int8_int16": 16, "int8_int8": 8}.get(dtype)
    return 0 if bits is None else max(0, min(31, 13 + int(math.log2(max(K, 1)) / 2) - bits + 3))


def draw(rng):
    while True:
        dtype, layout = rng.choice(_DTYPES), rng.choice(("row", "col"))
        family = rng.choice(("square", "general", "general", "few_rows", "few_rows", "narrow", "layer"))
        scale = 1.0
        if family == "layer":
            d = 256 * rng.randint(4, 16)
            ffn = 128 * round(d * 2.6875 / 128)
            M = _size(rng, 1, 2048)
            c = _layer("", dtype, M, d, ffn, layout, _shift(dtype, d))
        else:
            if family == "square":
                M = N = K = _size(rng, 256, 8192)
            elif family == "general":
                M, N, K = (_size(rng, 256, 8192) for _ in range(3))
            elif family == "few_rows":
                M, N, K, scale = _size(rng, 1, 256), _size(rng, 1024, 12288), _size(rng, 1024, 12288), 0.02
            else:
                M, N, K = _size(rng, 1024, 8192), _size(rng, 16, 128), _size(rng, 512, 8192)
            c = _gemm("", dtype, M, N, K, layout, scale, _shift(dtype, K))
        del c["name"]
        if sum(M * N * K for M, N, K in _shapes(c)) <= _MAX_MACS:
            return c


def _shapes(case):
    """(M, N, K) of the case's GEMMs."""
    if case["kind"] == "gemm":
        return [(case["M"], case["N"], case["K"])]
    M, d, ffn = case["M"], case["d"], case["ffn"]
    return [(M, 3 * d, d), (M, d, d), (M, ffn, d), (M, d, ffn)]


def _operands(case, seed):
    """[(M, N, K, A, B)] of the case, on the GPU, from the seed."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    col, int8 = case["layout"] == "col", case["dtype"] != "bf16"
    half = case["kind"] == "layer"
    ops = []
    for M, N, K in _shapes(case):
        b_shape = (N, K) if col else (K, N)
        if int8:
            A = torch.randint(-128, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8)
            lo, hi = (-64, 64) if half else (-128, 128)
            B = torch.randint(lo, hi, b_shape, generator=gen, device="cuda", dtype=torch.int8)
        else:
            A = torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16)
            B = torch.randn(b_shape, generator=gen, device="cuda").mul_(case["b_scale"]).to(torch.bfloat16)
        ops.append((M, N, K, A, B))
    return ops


def prepare(case, seed):
    layout = G.GEMM_B_COL_MAJOR_NxK if case["layout"] == "col" else G.GEMM_B_ROW_MAJOR_KxN
    calls = [(M, N, K, A, K, B, B.shape[1], layout, torch.empty((M, N), device="cuda", dtype=_OUT[case["dtype"]]), N)
             for M, N, K, A, B in _operands(case, seed)]
    return {"dtype": case["dtype"], "shift": case["shift"], "calls": calls}


def run(state):
    dtype = state["dtype"]
    out = []
    for args in state["calls"]:
        if dtype == "bf16":
            status = G.gemm_bf16_f32acc_bf16(*args)
        elif dtype == "int8":
            status = G.gemm_s8s8_s32(*args)
        elif dtype == "int8_int16":
            status = G.gemm_s8s8_s16(*args, state["shift"])
        else:
            status = G.gemm_s8s8_s8(*args, state["shift"])
        G.check(status)
        out.append(args[8])
    return out


def work(case):
    esize = 2 if case["dtype"] == "bf16" else 1
    osize = {"int8": 4, "int8_int16": 2, "int8_int8": 1, "bf16": 2}[case["dtype"]]
    shapes = _shapes(case)
    return {"bytes": sum(esize * (M * K + K * N) + osize * M * N for M, N, K in shapes),
            "flops": sum(2 * M * N * K for M, N, K in shapes)}


def exact(case, seed):
    out = []
    for M, N, K, A, B in _operands(case, seed):
        C = A.double() @ (B.double().t() if case["layout"] == "col" else B.double())
        if case["dtype"] == "int8":
            C = C.to(torch.int32)  # every int32 sum is exact in 64 bits
        elif case["dtype"] != "bf16":
            bits = 16 if case["dtype"] == "int8_int16" else 8
            C = torch.round(C / 2.0 ** case["shift"])  # ties to even
            C = C.clamp_(-2.0 ** (bits - 1), 2.0 ** (bits - 1) - 1).to(_OUT[case["dtype"]])
        out.append(C)
    return out
