"""The few-row kernel (at most 16 rows of A, or columns of B, against a
K-contiguous operand): every element against the oracle at the edges of its
strips (32 rows), batches (128 bytes of K), clusters and row groups (8), with
odd pitches and bases of the small operand and of C, at the int8 extremes, and
the plan query's route.  int8 is exact; bf16 is held to the library's bound
|C - ref| <= 2^-8 |ref| + 2^-20 sum |a b|, which one rounding to bf16 and an
fp32 sum in any order satisfy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_13282_gb300 import gemm as G
from paper_2512_13282_gb300 import workloads as W
from tests import gpu_util as U

COL = G.GEMM_B_COL_MAJOR_NxK


def _run(dtype, M, N, K, seed, shift=0, **kw):
    rnd = W.random_bf16 if dtype == "bf16" else W.random_int8
    A, B = rnd((M, K), seed), rnd((N, K), seed + 1)
    C = U.run(dtype, A, B, COL, shift=shift, **kw)
    if dtype == "bf16":
        ref, mag = oracle.gemm_bf16(A, B, COL)
        assert oracle.bf16_within_bound(C, ref, mag).all()
    else:
        want = oracle.gemm_s8(A, B, COL)
        if dtype != "int8":
            want = oracle.requantize(want, shift, 16 if dtype == "int8_int16" else 8)
        assert np.array_equal(C.astype(np.int64), want)


# rows of the small operand x rows of the large one x K
EDGES = [(1, 1, 16), (1, 33, 128), (7, 31, 144), (8, 32, 2048), (9, 64, 1040), (16, 95, 4112), (16, 129, 496),
         (3, 700, 16384), (13, 4100, 256)]


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("dtype", ["int8", "bf16", "int8_int8"])
@pytest.mark.parametrize("R,L,K", EDGES, ids=[f"{r}x{n}x{k}" for r, n, k in EDGES])
def test_few_rows(dtype, R, L, K):
    for M, N in ((R, L), (L, R)):
        st, plan = G.gemm_plan_query(M, N, K, dtype != "bf16", COL)
        narrow = dtype == "bf16" and M > 16 and K < 1024  # the tensor-core kernels' then
        assert st == 0 and (plan["route"] == G.GEMM_ROUTE_FEW_ROWS) == (not narrow)
        _run(dtype, M, N, K, seed=R + L + K, shift=7)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("K", [1, 15, 130, 1001])
def test_few_rows_ragged_k_and_odd_small_operand(dtype, K):
    """K that ends inside a 16-byte piece (the large operand's pitch rounded
    up to 16 bytes), the small operand and C on odd pitches and bases."""
    pad = (-K) % 16
    _run(dtype, 11, 70, K, seed=K, lda=K + 3, ldb=K + pad, ldc=75, a_off=1, c_off=1)
    _run(dtype, 70, 11, K, seed=K, lda=K + pad, ldb=K + 5, ldc=13, b_off=1, c_off=3)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("dtype,R,K,pad,off", [("int8", 16, 2048, 1, 0), ("int8", 9, 640, 2, 3), ("int8", 3, 1040, 4, 1),
                                               ("int8", 8, 512, 8, 0), ("int8", 1, 2064, 0, 2), ("bf16", 16, 1032, 1, 0),
                                               ("bf16", 8, 2048, 2, 3), ("bf16", 2, 1024, 4, 1), ("bf16", 1, 1544, 0, 1)])
def test_few_rows_small_operand_by_words(dtype, R, K, pad, off):
    """A small operand on every alignment that is not 16 bytes, over several
    batches: read by aligned words, at its first and last bytes element by
    element."""
    _run(dtype, R, 130, K, seed=K + R, lda=K + pad, a_off=off)
    _run(dtype, 1100, R, K, seed=K - R, ldb=K + pad, b_off=off)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
def test_few_rows_int8_extremes():
    """All -128 at the largest K (2147467264), and -128 x 127."""
    A, B = np.full((16, 131071), -128, np.int8), np.full((40, 131071), -128, np.int8)
    ld = 131072
    assert (U.run("int8", A, B, COL, ldb=ld) == 2147467264).all()
    assert (U.run("int8", B, A, COL, lda=ld) == 2147467264).all()
    B[:, :] = 127
    assert (U.run("int8", A, B, COL, ldb=ld) == -16256 * 131071).all()


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
def test_few_rows_nan_and_inf_stay_in_their_rows():
    """A NaN or infinity in a row of either operand reaches that row or
    column of C and no other (padding rows and columns repeat real ones)."""
    M, N, K = 5, 45, 300
    A, B = W.random_bf16((M, K), 3), W.random_bf16((N, K), 4)
    A[2, 299], B[44, 0] = 0x7FC0, 0x7F80  # NaN; +Inf
    C = torch.from_numpy(U.run("bf16", A, B, COL, ldb=304).view(np.int16).copy()).view(torch.bfloat16).float().numpy()
    bad = ~np.isfinite(C)
    assert np.isnan(C[2]).all() and bad[:, 44].all()
    bad[2], bad[:, 44] = False, False
    assert not bad.any()


def test_route_limits():
    """17 rows, a row-major B, an unaligned K pitch or a forced plan take
    the other kernels."""
    def route(M, N, K, int8, layout):
        return G.gemm_plan_query(M, N, K, int8, layout)[1]["route"]
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()
    few = G.GEMM_ROUTE_FEW_ROWS
    assert route(16, 4096, 4096, True, COL) == few and route(4096, 16, 4096, False, COL) == few
    assert route(17, 4096, 4096, True, COL) != few and route(4096, 17, 4096, False, COL) != few
    assert route(16, 4096, 4096, True, G.GEMM_B_ROW_MAJOR_KxN) != few
    assert route(16, 4096, 4097, False, COL) != few


def test_few_row_indexes_fit_an_int():
    """K up to INT32_MAX is accepted: the calls that the few-row kernel takes
    have every k index it forms (the cluster's slices and a round of batches
    past them) below 2^31, longer ones go elsewhere."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()
    for K in (1 << 20, 1 << 28, 1 << 30, (1 << 30) + 8, (1 << 31) - 512, (1 << 31) - 8):
        for M, N in ((2, 32), (16, 1000), (64, 8), (1, 1 << 20)):
            st, plan = G.gemm_plan_query(M, N, K, False, COL)
            assert st == G.GEMM_OK
            if plan["route"] == G.GEMM_ROUTE_FEW_ROWS:
                slice_ = -(-(-(-K // plan["splits"])) // 64) * 64
                assert plan["splits"] * slice_ + 4 * 64 + 32 < 1 << 31, (M, N, K)


def test_few_rows_of_a_long_k_go_where_it_is_split_further():
    """Few strips of the streamed operand and a long K: more blocks than a
    cluster's eight share it on the other kernels; clusters that do not all run
    at once are not chosen."""
    from paper_2512_13282_gb300 import build
    build.build()
    G.gemm_reload_overrides()

    def few(M, N, K, int8):
        st, plan = G.gemm_plan_query(M, N, K, int8, COL)
        assert st == G.GEMM_OK
        return plan["splits"] if plan["route"] == G.GEMM_ROUTE_FEW_ROWS else 0

    for M, N, K, int8, c in ((1, 32, 32768, False, 8), (1, 32, 65536, False, 0), (1, 600, 8192, False, 8),
                             (1, 600, 16384, False, 0), (4, 600, 16384, False, 8), (4, 600, 32768, False, 0),
                             (32, 1, 65536, False, 0), (600, 16, 16384, False, 8), (1, 2400, 65536, False, 8),
                             (4, 10000, 16384, False, 0), (1, 128, 32768, True, 8), (1, 128, 65536, True, 0),
                             (8, 600, 32768, True, 0), (16, 600, 65536, True, 8), (600, 4, 65536, True, 8),
                             (16, 4096, 4096, True, 4), (4, 2400, 8192, True, 7), (4, 2656, 8192, True, 6),
                             (16, 2400, 8192, False, 7), (4, 2400, 8192, False, 8),
                             (4, 11008, 4096, False, 1), (1, 11008, 4096, True, 1), (1, 12288, 4096, False, 1)):
        assert few(M, N, K, int8) == c, (M, N, K, int8)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("dtype,M,N,K", [("bf16", 2, 40, 40960), ("bf16", 5, 70, 24576), ("bf16", 70, 2, 24576), ("int8", 3, 70, 40960),
                                         ("int8", 7, 250, 24576), ("bf16", 16, 2400, 1024), ("int8", 4, 2656, 2048), ("int8", 9, 3200, 1040)])
def test_few_rows_around_the_long_k_limit(dtype, M, N, K):
    """Both sides of the limit, and clusters of 5 to 7 blocks."""
    _run(dtype, M, N, K, seed=M + K)
    _run(dtype, M, N, K - 32 * 1024 // 4 if K > 16384 else K + 16, seed=M - K)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("K", [32768, 40960])
def test_many_unaligned_rows_of_a_long_k(K):
    """More than 8 rows off the 16-byte grid: long slices go to other kernels."""
    before = G.gemm_launch_count()
    _run("int8", 13, 70, K, seed=K, lda=K + 8)
    assert (G.gemm_launch_count() - before == 1) == (K == 32768)


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("R", [3, 16])
@pytest.mark.parametrize("K,pad", [(271, 1), (500, 12), (1003, 5), (1009, 15), (2047, 1), (1030, 26)])
def test_few_rows_last_pieces(dtype, R, K, pad):
    """A K off the 16-byte grid: the last piece of a row is cut from what follows
    it, NaN and extremes there included, and the last row's ends at the matrix."""
    L = 70
    rng = np.random.default_rng(K)
    ld = K + pad

    def filled(rows):
        if dtype == "bf16":
            buf = np.full((rows, ld), 0x7FC0, np.uint16)  # NaN behind each row
            buf[:, :K] = W.random_bf16((rows, K), int(rng.integers(1 << 30)))
        else:
            buf = np.full((rows, ld), -128, np.int8)
            buf[:, :K] = W.random_int8((rows, K), int(rng.integers(1 << 30)))
        return buf

    A, B = filled(R), filled(L)
    for X, Y in ((A, B), (B, A)):
        M, N = X.shape[0], Y.shape[0]
        view = (lambda a: a.view(np.int16)) if dtype == "bf16" else (lambda a: a)
        tx, ty = torch.from_numpy(view(X)).cuda(), torch.from_numpy(view(Y)).cuda()
        c = torch.zeros((M, N), dtype=torch.int16 if dtype == "bf16" else torch.int32, device="cuda")
        fn = G.gemm_bf16_f32acc_bf16 if dtype == "bf16" else G.gemm_s8s8_s32
        G.gemm_reload_overrides()
        # the pitch of the small operand need not be a multiple of 16 bytes, the large one's is
        assert fn(M, N, K, tx, ld, ty, ld, COL, c, N) == G.GEMM_OK
        torch.cuda.synchronize()
        C = c.cpu().numpy()
        x, y = np.ascontiguousarray(X[:, :K]), np.ascontiguousarray(Y[:, :K])
        if dtype == "bf16":
            ref, mag = oracle.gemm_bf16(x, y, COL)
            assert oracle.bf16_within_bound(C.view(np.uint16), ref, mag).all()
        else:
            assert np.array_equal(C.astype(np.int64), oracle.gemm_s8(x, y, COL))


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("M", [1, 2, 8])
def test_few_rows_are_as_precise_as_the_kernels_before(M, monkeypatch):
    """The share of bf16 results that are not the nearest to the sum in 64 bits,
    against the kernel that takes the call otherwise (the CUDA cores for one and two
    rows, the tensor cores above): no larger, but for the noise of the counts."""
    gen = torch.Generator(device="cuda").manual_seed(M)
    off = {"": 0, str(min(M, 2) if M <= 2 else 2): 0}
    cells = 0
    for N, K in ((12288, 1024), (12288, 4096), (4096, 4096), (4096, 11008), (2048, 12288)):
        for _ in range(24 // M):
            A = torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16)
            B = torch.randn((N, K), generator=gen, device="cuda").to(torch.bfloat16)
            near = (A.double() @ B.double().t()).to(torch.bfloat16)
            cells += M * N
            for limit in off:
                if limit:
                    monkeypatch.setenv("GB300_GEMM_SKINNY_MAX_M", limit)
                else:
                    monkeypatch.delenv("GB300_GEMM_SKINNY_MAX_M", raising=False)
                G.gemm_reload_overrides()
                C = torch.empty((M, N), device="cuda", dtype=torch.bfloat16)
                assert G.gemm_bf16_f32acc_bf16(M, N, K, A, K, B, K, COL, C, N) == G.GEMM_OK
                off[limit] += int((C != near).sum())
    monkeypatch.undo()
    G.gemm_reload_overrides()
    rows, before = off.values()
    assert before > 0 and rows <= before + 4 * before ** 0.5, (rows, before, cells)
