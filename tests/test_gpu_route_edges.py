"""Edges of the routes: operands that are staged or re-pitched from odd bases
and pitches (whole 16-byte pieces are read by aligned words there, and the
first and last elements of a matrix must not be reached past), calls captured
into a CUDA graph on a stream that has no scratch yet, and the sizes where one
route ends and the next begins.  int8 is exact; bf16 is held to the library's
bound |C - ref| <= 2^-8 |ref| + 2^-20 sum |a b|."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_13282_gb300 import gemm as G
from paper_2512_13282_gb300 import workloads as W
from tests import gpu_util as U

ROW, COL = G.GEMM_B_ROW_MAJOR_KxN, G.GEMM_B_COL_MAJOR_NxK
needs_gpu = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")


def _operands(dtype, M, N, K, layout, seed):
    rnd = W.random_int8 if dtype == "int8" else W.random_bf16
    return rnd((M, K), seed), rnd((N, K) if layout == COL else (K, N), seed + 1)


def _check(dtype, A, B, layout, C):
    if dtype == "int8":
        assert np.array_equal(C.astype(np.int64), oracle.gemm_s8(A, B, layout))
    else:
        ref, mag = oracle.gemm_bf16(A, B, layout)
        assert oracle.bf16_within_bound(C, ref, mag).all()


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("layout", [ROW, COL])
@pytest.mark.parametrize("K,pad,off", [(577, 0, 0), (640, 0, 1), (641, 2, 3), (703, 0, 8), (705, 1, 13), (1016, 8, 5)])
def test_staged_from_odd_bases_and_pitches(dtype, layout, K, pad, off):
    M, N = 161, 203
    A, B = _operands(dtype, M, N, K, layout, K)
    C = U.run(dtype, A, B, layout, lda=K + pad, ldb=B.shape[1] + pad, a_off=off, b_off=off)
    _check(dtype, A, B, layout, C)


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype,M,N,K,layout", [
    ("int8", 512, 512, 512, COL), ("int8", 40, 300, 4000, ROW), ("int8", 6, 4096, 64, ROW),
    ("bf16", 256, 512, 3840, COL), ("bf16", 128, 4096, 4096, ROW), ("int8", 16, 4096, 4096, COL)])
def test_captured_on_a_stream_without_scratch(dtype, M, N, K, layout):
    G.gemm_reload_overrides()
    s = torch.cuda.Stream()
    A, B = _operands(dtype, M, N, K, layout, 9)
    view = (lambda x: x) if dtype == "int8" else (lambda x: x.view(np.int16))
    tA, tB = torch.from_numpy(view(A)).cuda(), torch.from_numpy(view(B)).cuda()
    tC = torch.zeros((M, N), dtype=torch.int32 if dtype == "int8" else torch.int16, device="cuda")
    fn = G.gemm_s8s8_s32 if dtype == "int8" else G.gemm_bf16_f32acc_bf16
    torch.cuda.synchronize()
    G.gemm_release_resources()
    # another stream's call loads the kernels; the captured stream has no scratch
    assert fn(M, N, K, tA, K, tB, B.shape[1], layout, tC, N, torch.cuda.default_stream()) == G.GEMM_OK
    torch.cuda.synchronize()
    tC.zero_()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        assert fn(M, N, K, tA, K, tB, B.shape[1], layout, tC, N, s) == G.GEMM_OK
    g.replay()
    torch.cuda.synchronize()
    C = tC.cpu().numpy()
    _check(dtype, A, B, layout, C if dtype == "int8" else C.view(np.uint16))


# C rows that allow no wide store leave row by row through the staging blocks:
# every tile width and family, partials with an odd pitch, a split tail
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["bf16", "int8", "int8_int16", "int8_int8"])
@pytest.mark.parametrize("bn,pair", [(64, 0), (96, 0), (128, 0), (128, 1), (192, 0), (192, 1), (224, 0), (224, 1), (256, 0),
                                     (256, 1)])
def test_odd_output_rows(monkeypatch, dtype, bn, pair):
    if dtype != "bf16" and bn < 128:
        pytest.skip("not compiled for int8")
    monkeypatch.setenv("GB300_GEMM_S8TM", "0")
    monkeypatch.setenv("GB300_GEMM_BN", str(bn))
    monkeypatch.setenv("GB300_GEMM_PAIR", str(pair))
    for M, N, K, ldc, off, extra in ((300, 259, 512, 261, 1, None), (513, 259, 1600, 259, 3, None),
                                     (200, 131, 2064, 133, 0, ("GB300_GEMM_SPLITS", "3")),
                                     (1300, 4099, 512, 4099, 0, ("GB300_GEMM_TAIL_SPLITS", "2"))):
        with monkeypatch.context() as m:
            if extra:
                m.setenv(*extra)
            kind = "bf16" if dtype == "bf16" else "int8"
            A, B = _operands(kind, M, N, K, COL, bn + M)
            C = U.run(dtype, A, B, COL, ldc=ldc, c_off=off, shift=9)
            if dtype in ("bf16", "int8"):
                _check(kind, A, B, COL, C)
            else:
                want = oracle.requantize(oracle.gemm_s8(A, B, COL), 9, 16 if dtype == "int8_int16" else 8)
                assert np.array_equal(C.astype(np.int64), want)


# the CUDA-core kernel with an unaligned column-major B, whose lanes read their
# pieces by aligned words inside the matrix
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("M,N,K,off", [(1, 33, 1001, 0), (2, 70, 515, 1), (2, 4, 17, 3), (1, 301, 4099, 5)])
def test_small_m_unaligned_column_major(dtype, M, N, K, off):
    A, B = _operands(dtype, M, N, K, COL, M + K)
    _check(dtype, A, B, COL, U.run(dtype, A, B, COL, b_off=off))


# 129 rows and more of the small operand: several Q tiles, one or more K
# splits, ragged edges of both operands; C stored by TMA or, with an odd pitch
# or base, element by element
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype,M,N,K,layout,kw", [
    ("int8", 129, 4096, 2048, COL, {}), ("int8", 129, 4096, 2048, ROW, {}), ("int8", 257, 2064, 4100, COL, {"ldb": 4112}),
    ("int8", 200, 3000, 4099, ROW, {"ldb": 3008, "ldc": 3001}), ("int8", 385, 12288, 1040, COL, {}),
    ("int8", 385, 8193, 2048, COL, {"ldc": 8193, "c_off": 1}), ("int8", 4096, 129, 2048, ROW, {}),
    ("int8", 3001, 200, 4096, COL, {}), ("int8", 2049, 300, 4096, ROW, {"ldc": 301}), ("int8", 8192, 520, 2064, COL, {}),
    ("int8_int16", 200, 4096, 4096, COL, {"shift": 9}), ("int8_int8", 192, 4096, 4096, ROW, {"shift": 14}),
    ("int8_int8", 4096, 200, 4096, COL, {"shift": 14}), ("int8_int16", 3001, 77, 4096, ROW, {"shift": 9}),
    ("int8_int8", 2000, 132, 4096, COL, {"shift": 13, "ldc": 133, "c_off": 1}),
    ("int8_int16", 8192, 520, 2064, ROW, {"shift": 8})])
def test_small_operand_kernel_with_several_tiles(dtype, M, N, K, layout, kw):
    rng = np.random.default_rng(M + N + K)
    A = rng.integers(-128, 128, (M, K), dtype=np.int8)
    B = rng.integers(-128, 128, (N, K) if layout == COL else (K, N), dtype=np.int8)
    A[-1], B[-1] = -128, -128
    # the query takes tight pitches: ask for the K or N that the call's pitch makes of it
    pk, pn = (kw.get("ldb", K), N) if layout == COL else (K, kw.get("ldb", N))
    st, plan = G.gemm_plan_query(M, pn, pk, True, layout)
    assert st == G.GEMM_OK and plan["route"] == G.GEMM_ROUTE_SMALL_OPERAND and plan["bn"] == 128
    C = U.run(dtype, A, B, layout, **kw)
    want = oracle.gemm_s8(A, B, layout)
    if dtype != "int8":
        want = oracle.requantize(want, kw["shift"], 16 if dtype == "int8_int16" else 8)
    assert np.array_equal(C.astype(np.int64), want)


def test_route_limits():
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()

    def route(M, N, K, int8, layout=ROW):
        st, plan = G.gemm_plan_query(M, N, K, int8, layout)
        assert st == G.GEMM_OK
        return plan["route"]

    # the one-launch int8 kernel: 2^24 multiply-adds and K = 512
    assert route(256, 256, 256, True) == G.GEMM_ROUTE_TINY and route(64, 512, 512, True) == G.GEMM_ROUTE_TINY
    assert route(256, 272, 256, True) != G.GEMM_ROUTE_TINY and route(64, 64, 513, True) != G.GEMM_ROUTE_TINY
    # the small-M kernel against the small-operand one, by what each has to move
    small_m, small_op = G.GEMM_ROUTE_SMALL_M, G.GEMM_ROUTE_SMALL_OPERAND
    assert [route(m, 4096, 4096, True) for m in (1, 2)] == [small_m, small_op]
    assert [route(m, 12288, 4096, True) for m in (2, 3)] == [small_m, small_op]
    assert [route(m, 2003, 3001, True) for m in (3, 4)] == [small_m, G.GEMM_ROUTE_TC_SINGLE]
    assert [route(m, 2003, 3001, True, COL) for m in (8, 17)] == [small_m, G.GEMM_ROUTE_TC_SINGLE]
    # several Q tiles of the small-operand kernel against the general path
    assert route(512, 4096, 4096, True, COL) == small_op and route(4096, 256, 4096, True) == small_op
    assert route(1024, 4096, 4096, True, COL) == G.GEMM_ROUTE_TC_PAIR and route(256, 1024, 1024, True) != small_op
    assert [route(m, 4096, 4096, False) for m in (2, 3)] == [small_m, G.GEMM_ROUTE_TC_SINGLE]


# how C is stored where TMA cannot: by the lanes where they can store whole
# words (two for 32-bit outputs) or C is a few columns or one block of rows
# tall, else row by row
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype,M,N,ldc,off,how", [
    ("bf16", 200, 130, 130, 0, "lanes"), ("bf16", 200, 130, 131, 0, "rows"), ("bf16", 200, 130, 130, 1, "rows"),
    ("int8_int16", 200, 130, 130, 0, "lanes"), ("int8_int16", 200, 130, 131, 0, "rows"),
    ("int8_int8", 200, 132, 132, 0, "lanes"), ("int8_int8", 200, 130, 130, 0, "rows"), ("int8_int8", 200, 132, 132, 2, "rows"),
    ("int8", 200, 130, 130, 0, "lanes"), ("int8", 200, 129, 129, 0, "rows"), ("int8", 200, 127, 127, 0, "lanes"),
    ("bf16", 65, 23, 23, 0, "lanes"), ("bf16", 65, 25, 25, 0, "rows"), ("bf16", 64, 131, 131, 0, "lanes"),
    ("bf16", 65, 131, 131, 0, "rows"), ("int8_int8", 65, 23, 23, 0, "lanes"), ("int8_int8", 64, 131, 131, 0, "lanes")])
def test_how_odd_output_rows_are_stored(monkeypatch, capfd, dtype, M, N, ldc, off, how):
    for var, v in (("S8TM", 0), ("TINY_MAX_MACS", 0), ("SPLITS", 1), ("DEBUG", 1)):
        monkeypatch.setenv("GB300_GEMM_" + var, str(v))
    kind = "bf16" if dtype == "bf16" else "int8"
    A, B = _operands(kind, M, N, 640, COL, M + N)
    capfd.readouterr()
    C = U.run(dtype, A, B, COL, ldc=ldc, c_off=off, shift=9)
    assert f"output by {how}" in capfd.readouterr().err
    if dtype in ("bf16", "int8"):
        _check(kind, A, B, COL, C)
    else:
        want = oracle.requantize(oracle.gemm_s8(A, B, COL), 9, 16 if dtype == "int8_int16" else 8)
        assert np.array_equal(C.astype(np.int64), want)


# the copies of operands with short rows: not much longer than the operand, and
# right at the ends of the rows and of the matrix, whose last pieces are read
# past the row where the matrix goes on
@pytest.mark.gpu
@needs_gpu
def test_short_rows_are_copied_at_their_length():
    M, N, K = 2_000_000, 24, 5
    A, B = W.random_bf16((M, K), 1), W.random_bf16((N, K), 2)
    tA, tB = (torch.from_numpy(x.view(np.int16)).cuda() for x in (A, B))
    tC = torch.zeros((M, N), dtype=torch.int16, device="cuda")
    G.gemm_release_resources()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert G.gemm_bf16_f32acc_bf16(M, N, K, tA, K, tB, K, COL, tC, N) == G.GEMM_OK
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert used < 5 * M * K * 2, used  # rows of 8 elements and a quarter to spare, not of 64
    C = tC.cpu().numpy().view(np.uint16)
    for rows in (slice(0, 300), slice(M - 300, M)):
        ref, mag = oracle.gemm_bf16(A[rows], B, COL)
        assert oracle.bf16_within_bound(C[rows], ref, mag).all()


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("K,pad,off", [(1, 0, 0), (7, 0, 1), (9, 1, 0), (21, 0, 3), (40, 0, 0), (47, 2, 1), (255, 0, 5),
                                       (300, 0, 0), (501, 3, 0), (513, 0, 7)])
def test_short_rows_staged(monkeypatch, dtype, K, pad, off):
    for var in ("S8TM", "TINY_MAX_MACS"):
        monkeypatch.setenv("GB300_GEMM_" + var, "0")
    M, N = 333, 77
    for layout in (ROW, COL):
        A, B = _operands(dtype, M, N, K, layout, K)
        C = U.run(dtype, A, B, layout, lda=K + pad, ldb=B.shape[1] + pad, a_off=off, b_off=off)
        _check(dtype, A, B, layout, C)


# the CUDA-core kernel reads aligned and unaligned column-major rows by code of
# its own each: the same sums, in the same order
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("M,N,K", [(1, 70, 2064), (2, 33, 4096), (5, 129, 1040), (8, 31, 527), (16, 64, 784)])
def test_small_m_aligned_and_unaligned_columns_agree(monkeypatch, dtype, M, N, K):
    monkeypatch.setenv("GB300_GEMM_SKINNY_MAX_M", "16")
    A, B = _operands(dtype, M, N, K, COL, M + N)
    C = U.run(dtype, A, B, COL, ldb=(K + 15) // 16 * 16)
    _check(dtype, A, B, COL, C)
    assert np.array_equal(C, U.run(dtype, A, B, COL, ldb=(K + 15) // 16 * 16 + 1, b_off=1))


# slices of A that fill the 48 KB of shared memory a kernel may use unasked
# (16 rows x 1536 bf16) or all but a little more
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("K", [1504, 1536, 1568, 3072])
def test_small_m_kernel_at_the_shared_memory_limit(monkeypatch, K):
    monkeypatch.setenv("GB300_GEMM_SKINNY_MAX_M", "16")
    # as many columns as give one slice of K per wave of blocks
    N = 32 * 608
    A, B = _operands("bf16", 12, N, K, COL, K)
    _check("bf16", A, B, COL, U.run("bf16", A, B, COL))


def test_small_m_limits():
    """The CUDA-core kernel keeps a B that the others would have to stage."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()

    def small(M, N, K, layout):
        st, plan = G.gemm_plan_query(M, N, K, True, layout)
        assert st == G.GEMM_OK
        return plan["route"] == G.GEMM_ROUTE_SMALL_M

    assert all(small(m, n, k, COL) for m in (3, 8) for n, k in ((12289, 4097), (9001, 16385), (20001, 20001)))
    assert [small(m, 5001, 5001, ROW) for m in (2, 3)] == [True, False]
    assert [small(m, 5, 700, ROW) for m in (4, 5)] == [True, False] and small(4, 33, 1500, ROW)
    assert small(8, 17, 3001, ROW) and not small(8, 65, 3001, ROW)
    assert small(8, 8200, 4288, ROW) and not small(8, 8204, 4288, ROW) and not small(8, 2008, 1500, ROW)


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "int8_int16", "int8_int8"])
@pytest.mark.parametrize("M,N,K,layout", [(8, 301, 4097, COL), (3, 4099, 2049, COL), (4, 5, 700, ROW), (8, 17, 3001, ROW), (4, 33, 1500, ROW),
                                          (2, 4096, 2048, ROW), (3, 2064, 1024, ROW), (4, 2064, 1024, ROW), (6, 1024, 1024, ROW),
                                          (7, 1024, 1024, ROW), (3, 1040, 8192, ROW)])
def test_small_m_limits_results(dtype, M, N, K, layout):
    A, B = _operands("int8", M, N, K, layout, M + N)
    C = U.run(dtype, A, B, layout, shift=10)
    want = oracle.gemm_s8(A, B, layout)
    if dtype != "int8":
        want = oracle.requantize(want, 10, 16 if dtype == "int8_int16" else 8)
    assert np.array_equal(C.astype(np.int64), want)


def test_tiny_limits():
    """The one-launch kernel beyond 2^24 multiply-adds: a short round of tiles, or
    rows off the 16-byte grid."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()

    def tiny(M, N, K, layout=ROW):
        st, plan = G.gemm_plan_query(M, N, K, True, layout)
        assert st == G.GEMM_OK
        return plan["route"] == G.GEMM_ROUTE_TINY

    assert tiny(128, 512, 512) and tiny(64, 1024, 512) and not tiny(64, 1040, 512) and not tiny(128, 512, 528)
    assert tiny(640, 89, 416) and tiny(511, 511, 129, COL) and tiny(511, 511, 385) and not tiny(511, 511, 386)
    assert tiny(1023, 511, 97) and not tiny(1025, 511, 97) and not tiny(1024, 512, 97 + 15) and not tiny(4001, 131, 127)
    assert tiny(512, 1257, 80) and tiny(1025, 511, 96) and not tiny(1023, 1023, 31)
    assert tiny(512, 512, 192) and not tiny(512, 512, 208) and not tiny(512, 528, 192)
    assert tiny(608, 1024, 96) and tiny(4800, 128, 64, COL) and not tiny(609, 1024, 64) and not tiny(608, 1024, 112)
    assert tiny(512, 608, 128) and not tiny(512, 624, 128) and not tiny(512, 608, 144)


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype", ["int8", "int8_int16", "int8_int8"])
@pytest.mark.parametrize("M,N,K,layout,pad,off", [(128, 512, 512, ROW, 0, 0), (640, 89, 416, COL, 0, 0), (511, 511, 385, ROW, 0, 1),
                                                  (1023, 511, 90, COL, 1, 3), (512, 512, 128, ROW, 4, 0), (512, 512, 384, ROW, 0, 0),
                                                  (512, 512, 192, COL, 0, 0), (384, 384, 512, ROW, 0, 0), (384, 400, 512, COL, 0, 0),
                                                  (608, 1024, 96, COL, 0, 0), (4800, 128, 64, ROW, 0, 0), (512, 608, 128, ROW, 0, 0),
                                                  (416, 512, 256, COL, 0, 0), (416, 528, 256, ROW, 0, 0)])
def test_tiny_limits_results(dtype, M, N, K, layout, pad, off):
    A, B = _operands("int8", M, N, K, layout, M + N)
    C = U.run(dtype, A, B, layout, lda=K + pad, ldb=B.shape[1] + pad, ldc=N + pad, a_off=off, c_off=off, shift=8)
    want = oracle.gemm_s8(A, B, layout)
    if dtype != "int8":
        want = oracle.requantize(want, 8, 16 if dtype == "int8_int16" else 8)
    assert np.array_equal(C.astype(np.int64), want)


# ... whose kernel for few rows would keep K-slice partials and counters
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype,M,N,K,layout", [
    ("int8", 6, 4096, 1024, ROW), ("int8", 1, 4096, 4096, ROW), ("int8", 3, 4099, 4099, COL), ("int8", 8, 17, 3001, ROW),
    ("bf16", 2, 4096, 4096, ROW), ("bf16", 1, 1024, 8192, ROW), ("bf16", 1, 64, 65536, COL), ("bf16", 5, 600, 32768, COL)])
def test_captured_few_rows_on_a_stream_without_scratch(dtype, M, N, K, layout):
    test_captured_on_a_stream_without_scratch(dtype, M, N, K, layout)


# narrow outputs through several tiles of the small-operand kernel (its choice
# depends on the output width; GB300_GEMM_DEBUG tells which kernel a call takes)
@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("dtype,M,N,K,layout,tiles,splits,kw", [
    ("int8_int16", 300, 12288, 4096, COL, (96, 3), 1, {"shift": 9}), ("int8_int8", 12288, 280, 4096, ROW, (96, 3), 1, {"shift": 14}),
    ("int8_int8", 300, 12280, 4096, COL, (96, 3), 1, {"shift": 14, "ldc": 12281, "c_off": 1}),
    ("int8_int16", 200, 4096, 4096, COL, (32, 2), 2, {"shift": 9, "ldc": 4099})])
def test_narrow_outputs_of_several_small_operand_tiles(monkeypatch, capfd, dtype, M, N, K, layout, tiles, splits, kw):
    monkeypatch.setenv("GB300_GEMM_DEBUG", "1")
    A, B = _operands("int8", M, N, K, layout, M)
    capfd.readouterr()
    C = U.run(dtype, A, B, layout, **kw)
    assert f"small operand: {tiles[0]} x {tiles[1]} tiles of 128 x 128, {splits} splits" in capfd.readouterr().err
    want = oracle.requantize(oracle.gemm_s8(A, B, layout), kw["shift"], 16 if dtype == "int8_int16" else 8)
    assert np.array_equal(C.astype(np.int64), want)


@pytest.mark.gpu
@needs_gpu
@pytest.mark.parametrize("M,N,K,layout,kw", [(7978, 321, 640, ROW, {}), (2048, 300, 4096, COL, {"ldc": 301}), (321, 4097, 2048, COL, {}),
                                             (4096, 201, 4096, ROW, {"c_off": 1}), (3000, 131, 2048, ROW, {})])
def test_small_operand_int32_rows_off_the_grid(M, N, K, layout, kw):
    """C that TMA cannot write: whichever kernel its stores leave the faster one."""
    A, B = _operands("int8", M, N, K, layout, M + N)
    _check("int8", A, B, layout, U.run("int8", A, B, layout, **kw))
