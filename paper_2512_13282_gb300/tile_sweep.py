"""Measure every forced tile plan of the tensor-core GEMM kernels on one GPU.

This is the measurement half of the balanced-point search (Sec. 4.5: the
starting values and each step's efficiency are measured on the device).  For
each shape of a fixed set -- the tensor-core GEMMs of the benchmark
workloads and a seeded sample of the roofline sweep sizes -- every plan the
library can be forced into (kernel family: one CTA per 128-row tile or a CTA
pair per 256-row tile; tile width BN; split-K factor S; split tail T) is timed
as a program runs it: calls back to back on one stream, over enough operand
copies that together they exceed L2 (up to 16), between two CUDA events around
at least `ms` milliseconds of calls, the median of three such runs after one
untimed.  Runs that long are under the power limit where a program's would be
(a burst of 8192^3 GEMMs runs 6 % faster than a stream of them, and favours
tiles that multiply more padding).  The result is written as JSON;
tile_model.py fits the planner's cost table to it.

    python -m paper_2512_13282_gb300.tile_sweep OUT.json [--ms 4] [--sample 60]

Needs a GPU and the built library.  Results of int8 GEMMs are exact whatever
the plan, and bf16 results differ only in summation order, so no plan is
checked here; the GPU tests cover every family, width and split.
"""
from __future__ import annotations

import argparse
import json
import os
import sys
import time

import numpy as np

from . import workloads as W
from .tile_model import candidate_plans, GB300

ENV_KEYS = ("GB300_GEMM_BN", "GB300_GEMM_PAIR", "GB300_GEMM_SPLITS", "GB300_GEMM_TAIL_SPLITS",
            "GB300_GEMM_SKINNY_MAX_M", "GB300_GEMM_S8TM", "GB300_GEMM_TINY_MAX_MACS")
# every int8 GEMM of the sweep on the tensor-core kernels
TC_ONLY = {"GB300_GEMM_SKINNY_MAX_M": 0, "GB300_GEMM_S8TM": 0, "GB300_GEMM_TINY_MAX_MACS": 0}


def sweep_shapes(sample: int = 60, seed: int = 11):
    """(M, N, K, dtype, layout) of the sweep: the workloads' GEMMs with M > 8
    that the tensor-core kernels run (int8-int32 and bf16), then `sample`
    roofline sizes (both dtypes, B column- and row-major in turn) drawn with
    `seed`, and half as many sizes that no tile divides (multiples of 16,
    uniform in log size from 128 to 8192, one dtype each)."""
    seen, out = set(), []
    for wl in ("square_sweep_512_4096", "square_8192", "transformer_projections", "irregular_skinny",
               "int8_square_256"):
        for g in W.WORKLOADS[wl].gemms:
            if g.M <= 8 or g.dtype not in ("int8", "bf16"):
                continue
            key = (g.M, g.N, g.K, g.dtype, g.layout)
            if key not in seen:
                seen.add(key)
                out.append(key)
    rng = np.random.default_rng(seed)
    sizes = W.roofline_sweep_sizes()
    for n, i in enumerate(rng.choice(len(sizes), sample, replace=False)):
        M, N, K = sizes[int(i)]
        for dt in ("int8", "bf16"):
            key = (M, N, K, dt, W.B_ROW_MAJOR if n % 3 == 2 else W.B_COL_MAJOR)
            if key not in seen:
                seen.add(key)
                out.append(key)
    for n in range(sample // 2):
        M, N, K = (16 * int(round(np.exp(rng.uniform(np.log(8), np.log(512))))) for _ in range(3))
        key = (M, N, K, "int8" if n % 2 else "bf16", W.B_ROW_MAJOR if n % 4 >= 2 else W.B_COL_MAJOR)
        if key not in seen and M * N * K <= 1 << 38:
            seen.add(key)
            out.append(key)
    return out


def main(argv=None):
    import torch

    from . import build as Bld
    from . import gemm as G

    ap = argparse.ArgumentParser()
    ap.add_argument("out")
    ap.add_argument("--ms", type=float, default=4.0)
    ap.add_argument("--sample", type=int, default=60)
    args = ap.parse_args(argv)
    Bld.build()
    G.library()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    st = torch.cuda.current_stream()
    shapes = sweep_shapes(args.sample)

    def operands(M, N, K, dtype, layout):
        """Copies of (A, B, C) that together exceed three times L2, at most 16."""
        b_shape = (K, N) if layout == W.B_ROW_MAJOR else (N, K)
        esize = 1 if dtype == "int8" else 2
        copies = []
        for i in range(max(2, min(16, -(-400_000_000 // (esize * (M * K + N * K)))))):
            gen = torch.Generator(device="cuda").manual_seed(31 + i)
            if dtype == "int8":
                A, B = (torch.randint(-128, 128, s, generator=gen, device=dev, dtype=torch.int8)
                        for s in ((M, K), b_shape))
            else:
                A, B = (torch.randn(s, generator=gen, device=dev).to(torch.bfloat16) for s in ((M, K), b_shape))
            copies.append((A, B, torch.empty((M, N), device=dev, dtype=torch.int32 if dtype == "int8" else torch.bfloat16)))
        return copies

    def setenv(d):
        for k in ENV_KEYS:
            os.environ.pop(k, None)
        for k, v in d.items():
            os.environ[k] = str(v)
        G.gemm_reload_overrides()

    def time_plan(M, N, K, dtype, layout, copies):
        ldb = N if layout == W.B_ROW_MAJOR else K
        fn = G.gemm_s8s8_s32 if dtype == "int8" else G.gemm_bf16_f32acc_bf16

        def calls(n):
            for i in range(n):
                A, B, C = copies[i % len(copies)]
                rc = fn(M, N, K, A, K, B, ldb, layout, C, N, st.cuda_stream)
                if rc != 0:
                    raise RuntimeError(f"{dtype} {M}x{N}x{K}: {G.gemm_status_string(rc)}")

        est = max(4e-6, 2.0 * M * N * K / 1.5e15)
        n = max(4, int(args.ms * 1e-3 / est))
        times = []
        for r in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(st)
            calls(n)
            b.record(st)
            torch.cuda.synchronize()
            if r:
                times.append(a.elapsed_time(b) * 1e3 / n)
        return sorted(times)[1]

    rows = []
    t0 = time.time()
    for (M, N, K, dtype, layout) in shapes:
        setenv(TC_ONLY)
        copies = operands(M, N, K, dtype, layout)
        default_us = time_plan(M, N, K, dtype, layout, copies)
        plans = []
        for c in candidate_plans(M, N, K, dtype, layout == W.B_COL_MAJOR, sms=sms, pair_slots=GB300["pair_slots"]):
            setenv(dict(TC_ONLY, GB300_GEMM_PAIR=int(c["pair"]), GB300_GEMM_BN=c["bn"],
                        GB300_GEMM_SPLITS=c["splits"], GB300_GEMM_TAIL_SPLITS=c["tail_splits"]))
            plans.append(dict(c, us=round(time_plan(M, N, K, dtype, layout, copies), 3)))
        best = min(plans, key=lambda p: p["us"])
        print(f"{dtype:4s} {M}x{N}x{K} {'col' if layout else 'row'}: planner {default_us:8.1f} us, best forced "
              f"{best['us']:8.1f} ({'pair' if best['pair'] else 'single'} BN={best['bn']} S={best['splits']} "
              f"T={best['tail_splits']})",
              file=sys.stderr, flush=True)
        rows.append({"M": M, "N": N, "K": K, "dtype": dtype, "layout": "col" if layout else "row",
                     "planner_us": round(default_us, 3), "plans": plans})
    setenv({})
    with open(args.out, "w") as f:
        json.dump({"device": torch.cuda.get_device_name(dev), "sms": sms, "ms": args.ms,
                   "method": "calls back to back over operand copies larger than L2", "statistic": "median of three runs",
                   "seconds": round(time.time() - t0, 1),
                   "shapes": rows}, f, indent=0)


if __name__ == "__main__":
    main()
