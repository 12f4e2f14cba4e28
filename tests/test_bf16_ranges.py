"""The K ranges of a bf16 GEMM on the tensor cores: they depend on its sizes
alone, and the kernels that sum them in registers give the bits of the split-K
partials and their reduction, on every tile width and output path."""
import random

import numpy as np
import pytest
import torch

import oracle
from paper_2512_13282_gb300 import gemm as G
from paper_2512_13282_gb300 import tile_model as T
from paper_2512_13282_gb300 import workloads as W
from tests import gpu_util as U

ROW, COL = G.GEMM_B_ROW_MAJOR_KxN, G.GEMM_B_COL_MAJOR_NxK


def test_ranges_are_a_property_of_the_sizes():
    """Two ranges of 2048 for the wide GEMMs of a 128-row layer, four and six
    for the others, as split-K partials or unsplit on a tile of at most 128
    columns; no plan sums other ranges."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()
    for N, K, r in ((12288, 4096, 2), (4096, 4096, 4), (11008, 4096, 2), (4096, 11008, 6)):
        assert T.sum_ranges(128, N, K, True) == r
    rng = random.Random(2)
    for _ in range(400):
        M, N, K = (int(2 ** rng.uniform(5, hi)) for hi in (11, 13, 13.5))
        layout = rng.randint(0, 1)
        st, plan = G.gemm_plan_query(M, N, K, False, layout)
        r = T.sum_ranges(M, N, K, layout == COL)
        assert st == G.GEMM_OK and plan["splits"] in (1, r)
        if r > 1 and plan["splits"] == 1:
            assert plan["bn"] <= T.MAX_SLAB_BN and plan["tail_splits"] == 0


# planned unsplit with several ranges: 64, 96 and 128 columns on one CTA, 128 on
# a pair, both layouts, last ranges and edges ragged
CASES = [(99, 24, 1045, ROW, 64), (18, 79, 1137, COL, 64), (131, 5489, 2880, COL, 96), (273, 5007, 5184, ROW, 128),
         (280, 4908, 4288, COL, 128), (137, 5025, 3072, ROW, -128), (692, 2541, 4480, COL, -128)]


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("kw", [{}, {"ldc": 3}, {"ldc": 4}], ids=["tight", "odd", "four"])
@pytest.mark.parametrize("M,N,K,layout,bn", CASES, ids=[f"{m}x{n}x{k}" for m, n, k, _, _ in CASES])
def test_ranges_in_registers_equal_split_k(M, N, K, layout, bn, kw, monkeypatch):
    for v in ("GB300_GEMM_SPLITS", "GB300_GEMM_BN", "GB300_GEMM_PAIR"):
        monkeypatch.delenv(v, raising=False)
    G.gemm_reload_overrides()
    st, plan = G.gemm_plan_query(M, N, K, False, layout)
    r = T.sum_ranges(M, N, K, layout == COL)
    assert r > 1 and (plan["splits"], plan["bn"], plan["route"]) == (
        1, abs(bn), G.GEMM_ROUTE_TC_PAIR if bn < 0 else G.GEMM_ROUTE_TC_SINGLE)
    A, B = W.random_bf16((M, K), M + K), W.random_bf16((N, K) if layout == COL else (K, N), N)
    A[M // 2, K - 1] = 0x7F80  # an infinity in the last range of one row
    # aligned output rows go through TMA, odd ones row by row, 8-byte ones by their lanes
    ldc = (N + 7) // 8 * 8 + kw["ldc"] if kw else N
    C = U.run("bf16", A, B, layout, ldc=ldc)
    monkeypatch.setenv("GB300_GEMM_SPLITS", str(r))
    want = U.run("bf16", A, B, layout, ldc=ldc)
    assert np.array_equal(C, want)
    rows = np.arange(M) != M // 2
    ref, mag = oracle.gemm_bf16(A[rows], B, layout)
    assert oracle.bf16_within_bound(C[rows], ref, mag).all()


def test_split_tails_are_a_property_of_the_sizes():
    """A split tail, with the tiles it covers, belongs to the ranges too: it
    stands as the fixed costs choose it, and no other plan gets one."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()
    for M, N, K, layout, bn, pair, tails in ((1072, 4848, 6800, COL, 256, True, 4), (8192, 1072, 4304, COL, 256, True, 5),
                                             (992, 7632, 8000, ROW, None, None, 0)):
        st, plan = G.gemm_plan_query(M, N, K, False, layout)
        assert st == G.GEMM_OK and plan["tail_splits"] == tails
        if tails:
            assert plan["bn"] == bn and (plan["route"] == G.GEMM_ROUTE_TC_PAIR) == pair
    rng = random.Random(4)
    for _ in range(400):
        M, N, K = (int(2 ** rng.uniform(9, 13)) for _ in range(3))
        layout = rng.randint(0, 1)
        st, plan = G.gemm_plan_query(M, N, K, False, layout)
        want = T.range_plan(M, N, K, layout == COL)
        assert st == G.GEMM_OK and plan["tail_splits"] == want["tail_splits"]
        if want["tail_splits"]:
            assert (plan["bn"], plan["route"] == G.GEMM_ROUTE_TC_PAIR) == (want["bn"], want["pair"])


def test_small_a_takes_long_steps():
    """Few rows with an A below 128 KB: fewer CTAs and longer K steps than for
    the same tiles with a larger A; the ranges stay."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()
    for M, N, K in ((14, 12368, 2576), (6, 8960, 1705), (6, 11008, 2048)):
        st, few = G.gemm_plan_query(M, N, K, False, ROW)
        assert st == G.GEMM_OK and few["splits"] == T.sum_ranges(M, N, K, False) == 3
    st, many = G.gemm_plan_query(32, 12368, 2576, False, ROW)
    assert st == G.GEMM_OK and many["splits"] == 1 and T.sum_ranges(32, 12368, 2576, False) == 3
