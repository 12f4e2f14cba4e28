// gemm_rows.cu -- GEMMs with one operand of at most 16 rows against an
// operand whose rows are K contiguous (a decode batch or one token against
// weights stored N x K, a tall matrix against a narrow weight): the large
// operand W goes from HBM into registers that already are operands of warp
// matrix instructions.
//
// With so few rows the time is the time to read W once, plus whatever the
// kernel spends before its first and after its last byte.  The tcgen05
// kernels pass every byte through a shared-memory ring (and, for int8,
// through converter warps and tensor memory) and pay those hand-offs per
// k-block; here a lane loads 16 bytes of W and multiplies them:
//
//   - W is the 16-row A operand of mma.sync m16n8k16, X (the small operand)
//     the 8-column B operand, so X costs ceil(rows / 8) instructions per
//     16 x 16 of W.
//   - The sum over k does not depend on its order, so the four k slots a
//     lane (g = lane / 4, q = lane % 4) holds of a k16 step are given four
//     consecutive k of its own 16 bytes, and X is read at the same k: W's
//     registers are MMA operands as they are loaded, without a shuffle.
//   - int8: a byte b becomes the fp16 1024 + (b + 128) by placing it under
//     the exponent of 1024, and one packed subtraction of 1152 leaves b
//     exactly (five instructions per four values); products are at most
//     2^14 and an accumulator takes at most 512 of them before it is added
//     to int32, so every fp32 sum is an integer of at most 2^23, exact.
//
// A block of four warps owns 32 rows of W and a K slice; the warps take
// 128-byte deep batches of the slice in turn and are summed in warp order (one or
// two bf16 rows pairwise) in shared memory.  K is split over the blocks of a cluster (1-8), whose sums
// meet in distributed shared memory in rank order: results do not depend on
// scheduling, and there are no partials in global memory, no counters and no
// second launch.  Each half of a batch is reloaded as soon as it has been
// multiplied, so that a lane keeps about 128 bytes in flight.  A block asks
// for its first batches in L2 before it waits for the previous kernel of the
// stream (a prefetch reads nothing into the block, so it does not matter
// whether that kernel still writes W).
//
// What bounds it: the HBM stream (5.0-5.6 TB/s of W on 100 MB) and, for the
// smaller calls, the ~3 us from launch to last store.  Measured on GB300,
// calls back to back on operands larger than L2, against the kernel that took
// the shape before (B stored N x K, K = 4096 unless given): int8 16 x 12288
// 17.7 -> 13.2 us, 16 x 4096 10.4 -> 6.7, 8 x 12288 28.0 -> 11.7, 1 x 12288
// 15.2 -> 11.4, 16 x 2048 x 2048 25.4 -> 4.1; bf16 1 x 12288 26.4 -> 19.1,
// 1 x 4096 x 11008 19.5 -> 16.7, 1 x 4096 10.9 -> 7.4, 16 x 12288 21.8 ->
// 20.0, 16 x 4096 10.9 -> 8.5.
// Tried: W through a TMA ring with 16 warps (bound by the latency of X and of
// the consumers, 18-32 us for 16 x 12288), cp.async queues in shared memory
// (130 KB in flight per SM; 1-3 us slower below 8 rows), and W stored K x N
// (four k-rows a lane; slower than the CUDA-core kernel at one row and than
// the tensor-core kernels above).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "gemm_internal.h"

namespace gb300 {

namespace {

constexpr int kRowsWarps = 4;
constexpr int kRowsThreads = kRowsWarps * 32;
constexpr int kStrip = 32;  // rows of W per block
// words per row of the shared sums: the accumulators' lanes store to it
// without bank conflicts
constexpr int kSumPitch = 36;
// Resident blocks per SM: 4 (at most 128 registers a thread; 5 measured no
// faster), and 5 for bf16 against 8 rows, which fits in 96.
constexpr int kRowsBlocks = 4;
template <int NT, bool INT8>
constexpr int rows_blocks() {
  return NT == 1 && !INT8 ? 5 : kRowsBlocks;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The 32-bit word at the same shared-memory offset in block `rank` of the cluster.
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr, uint32_t rank) {
  uint32_t a, v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

template <bool INT8>
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  if constexpr (INT8)
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  else
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The 16 bytes at a, of which the first `valid` are read (element by element
// of `es` bytes) and the rest are zero.  Out of line: the ends of W's and X's
// rows.
__device__ __noinline__ uint4 load16_edge(const uint8_t *a, int es, int valid) {
  uint32_t w[4] = {0u, 0u, 0u, 0u};
  for (int i = 0; i < 16 && i < valid; i += es) {
    const uint32_t v =
        es == 1 ? (uint32_t)__ldg(a + i) : (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(a + i));
    const uint32_t b = v << (8 * (i & 3));
    w[0] |= i < 4 ? b : 0u, w[1] |= i >> 2 == 1 ? b : 0u, w[2] |= i >> 2 == 2 ? b : 0u, w[3] |= i >> 2 == 3 ? b : 0u;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void store_out(const RowsParams &p, bool int8, int64_t at, uint32_t v) {
  if (!int8) {
    const __nv_bfloat16 h = __float2bfloat16_rn(__uint_as_float(v));
    reinterpret_cast<uint16_t *>(p.C)[at] = *reinterpret_cast<const uint16_t *>(&h);
  } else if (p.out_bits == 32) {
    reinterpret_cast<int32_t *>(p.C)[at] = (int32_t)v;
  } else {
    const int32_t hi = (1 << (p.out_bits - 1)) - 1, lo = -hi - 1;
    const int32_t q = requantize_s32((int32_t)v, p.out_shift, lo, hi);
    if (p.out_bits == 16)
      reinterpret_cast<int16_t *>(p.C)[at] = (int16_t)q;
    else
      reinterpret_cast<int8_t *>(p.C)[at] = (int8_t)q;
  }
}

// The 16 bytes at a, on any boundary of X = [lo, hi), as four or five aligned
// words, shifted (X on odd addresses): element by element they took longer
// than the stream (odd X pitch, element by element / this: bf16 4 x 12288 x 4096
// 51.3 / 23.0 us, 16 x 4096 x 4096 29.8 / 12.5, int8 4 x
// 4096 x 4096 14.5 / 8.1, 16 x 4096 x 4096 26.5 / 10.3).
__device__ __forceinline__ uint4 load16_words(const uint8_t *a, const uint8_t *lo, const uint8_t *hi, int es) {
  const uint32_t off = (uint32_t)reinterpret_cast<uintptr_t>(a) & 3u, sh = 8u * off;
  const uint8_t *al = a - off;
  if (al < lo || al + (off ? 20 : 16) > hi) return load16_edge(a, es, 16);
  const uint32_t *q = reinterpret_cast<const uint32_t *>(al);
  const uint32_t w0 = __ldg(q), w1 = __ldg(q + 1), w2 = __ldg(q + 2), w3 = __ldg(q + 3), w4 = off ? __ldg(q + 4) : 0u;
  return make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh),
                    __funnelshift_r(w3, w4, sh));
}

// The same of a row in [lo, hi): a row's last, partial piece is read whole and cut
// where the matrix goes on behind it, element by element only at its end (element
// by element everywhere it took as long as the rest of a small call: int8 16 x 64 x
// 271 8.7 us, 3.1 for K = 256).  Out of line for int8 against 16 rows, whose loop
// it cost 6 % inlined (16 x 11008 x 4096 14.6 us, 13.5 out of line); inlined
// elsewhere, where the call costs small calls 0.5 us.
__device__ __forceinline__ uint4 load16_part(const uint8_t *a, const uint8_t *lo, const uint8_t *hi, int es, int valid) {
  if (a + 16 > hi) return load16_edge(a, es, valid);
  const uint4 v = (reinterpret_cast<uintptr_t>(a) & 15u) == 0 ? __ldg(reinterpret_cast<const uint4 *>(a))
                                                               : load16_words(a, lo, hi, es);
  auto keep = [&](uint32_t w, int at) {
    const int n = valid - at;
    return n >= 4 ? w : n <= 0 ? 0u : w & (0xffffffffu >> (32 - 8 * n));
  };
  return make_uint4(keep(v.x, 0), keep(v.y, 4), keep(v.z, 8), keep(v.w, 12));
}

__device__ __noinline__ uint4 load16_part_call(const uint8_t *a, const uint8_t *lo, const uint8_t *hi, int es, int valid) {
  return load16_part(a, lo, hi, es, valid);
}

// NT: 8-row groups of X.  XVEC: X's rows start on 16-byte boundaries (a kernel
// of its own for those that do not, whose loads need more registers).
//
// FINE: one or two rows of X in bf16.  An MMA leaves its fp32 sum truncated, and
// one chain of MMAs over a warp's share of K was further off than the fp32 FMAs of
// the CUDA-core kernel that took those rows before: 0.035 % of the results were
// not the nearest bf16 against 0.009 % (K = 1024 to 12288; for 4 to 16 rows, where
// the other choice is the tensor cores, 0.033 against 0.062).  Here a chain ends
// with its batch (four MMAs), four batches are added in fp32 and their sums again:
// 0.0102 % of 13.2 M results, 0.0099 on the CUDA cores, in the same time (1 x 12288
// x 4096 19.1 us).  (Compensated sums, or chains spread over MMA columns that
// multiply zeros, would make NaN of infinities.)
template <int NT, bool INT8, bool XVEC, bool FINE>
__global__ void __launch_bounds__(kRowsThreads, rows_blocks<NT, INT8>()) gemm_rows_kernel(const RowsParams p) {
  constexpr int ES = INT8 ? 1 : 2;
  constexpr int kHalf = 64 / ES;       // k per half batch: 64 bytes of each row, 16 a lane
  constexpr int kBatch = 2 * kHalf;
  // batches after which an accumulator holds 512 products; FINE: that are added up
  constexpr int kFlush = INT8 ? 512 / kBatch : 4;
  static_assert(!FINE || (NT == 1 && !INT8), "one or two bf16 rows");
  extern __shared__ __align__(16) uint32_t red[];  // [warp][row of X][row of W], then the block's sums
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const uint32_t rank = p.cluster > 1 ? cluster_rank() : 0u;
  const int64_t n0 = (int64_t)(blockIdx.x / p.cluster) * kStrip;
  const int kbeg = (int)rank * p.kslice;
  const int kend = min(p.K, kbeg + p.kslice);  // kbeg < kend (rows_geometry), no overflow (kRowsMaxK)
  const int nb = (kend - kbeg + kBatch - 1) / kBatch;
  const int64_t pitch = p.ldw * ES;
  const int R = p.R;

  // The lane's bytes of a half batch: 16 q .. of W's rows n0 + 8 i + g and of
  // X's rows 8 j + g.  Rows past the last repeat another: their sums are not
  // stored.
  const uint8_t *wp[4], *xp[NT];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t n = n0 + 8 * i + g;
    wp[i] = static_cast<const uint8_t *>(p.W) + (n < p.NW ? n : p.NW - 1) * pitch + 16 * q;
  }
#pragma unroll
  for (int j = 0; j < NT; ++j)
    xp[j] = static_cast<const uint8_t *>(p.X) + (8 * j + g < R ? 8 * j + g : 0) * p.ldx * ES + 16 * q;
  const uint8_t *x_lo = static_cast<const uint8_t *>(p.X), *x_hi = x_lo + ((R - 1) * p.ldx + p.K) * ES;

  griddep_launch_dependents();
  {  // the warp's first batch: 128 bytes of row n0 + lane
    const int64_t n = n0 + lane, k = kbeg + warp * kBatch;
    if (n < p.NW && k < kend) prefetch_l2(static_cast<const uint8_t *>(p.W) + n * pitch + k * ES);
  }
  griddep_wait();

  auto load_part = [&](const uint8_t *a, const uint8_t *lo, const uint8_t *hi, int valid) {
    return INT8 && NT == 2 ? load16_part_call(a, lo, hi, ES, valid) : load16_part(a, lo, hi, ES, valid);
  };
  auto load_half = [&](int k, uint4 (&w)[4], uint4 (&x)[NT]) {
    const int64_t at = (int64_t)k * ES;
    const int valid = (kend - k) * ES - 16 * q;  // bytes of the lane's piece before the slice's end
    const bool whole = valid >= 16;
    if (whole) {
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = __ldcs(reinterpret_cast<const uint4 *>(wp[i] + at));
    } else if (valid <= 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = make_uint4(0u, 0u, 0u, 0u);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        w[i] = load_part(wp[i] + at, static_cast<const uint8_t *>(p.W),
                         static_cast<const uint8_t *>(p.W) + (p.NW - 1) * pitch + (int64_t)p.K * ES, valid);
    }
    if (valid <= 0) {
#pragma unroll
      for (int j = 0; j < NT; ++j) x[j] = make_uint4(0u, 0u, 0u, 0u);
    } else if (whole && XVEC) {
#pragma unroll
      for (int j = 0; j < NT; ++j) x[j] = __ldg(reinterpret_cast<const uint4 *>(xp[j] + at));
    } else if (whole) {
#pragma unroll
      for (int j = 0; j < NT; ++j) x[j] = load16_words(xp[j] + at, x_lo, x_hi, ES);
    } else {
#pragma unroll
      for (int j = 0; j < NT; ++j) x[j] = load_part(xp[j] + at, x_lo, x_hi, valid);
    }
  };

  float acc[2][NT][4];
  int32_t iacc[INT8 ? 2 : 1][NT][4];  // int8: the exact sums so far
  float near[FINE ? 2 : 1][NT][4], far[FINE ? 2 : 1][NT][4];  // FINE: the sums of up to kFlush batches, and of those
  auto each = [&](auto &&f) {
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) f(t, j, e);
  };
  each([&](int t, int j, int e) {
    acc[t][j][e] = 0.f;
    if constexpr (INT8) iacc[t][j][e] = 0;
    if constexpr (FINE) near[t][j][e] = far[t][j][e] = 0.f;
  });

  auto multiply = [&](const uint4 (&w)[4], const uint4 (&x)[NT]) {
    uint32_t wr[4][4], xr[NT][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) wr[i][0] = w[i].x, wr[i][1] = w[i].y, wr[i][2] = w[i].z, wr[i][3] = w[i].w;
#pragma unroll
    for (int j = 0; j < NT; ++j) xr[j][0] = x[j].x, xr[j][1] = x[j].y, xr[j][2] = x[j].z, xr[j][3] = x[j].w;
    if constexpr (!INT8) {
#pragma unroll
      for (int i = 0; i < 2; ++i)  // four of the lane's 8 k
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int j = 0; j < NT; ++j)
            mma16816<INT8>(acc[t][j], wr[2 * t][2 * i], wr[2 * t + 1][2 * i], wr[2 * t][2 * i + 1],
                           wr[2 * t + 1][2 * i + 1], xr[j][2 * i], xr[j][2 * i + 1]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {  // four of the lane's 16 k
        uint32_t b[NT][2];
#pragma unroll
        for (int j = 0; j < NT; ++j) s8x4_to_f16x4(xr[j][i], b[j][0], b[j][1]);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          uint32_t a[4];
          s8x4_to_f16x4(wr[2 * t][i], a[0], a[2]);
          s8x4_to_f16x4(wr[2 * t + 1][i], a[1], a[3]);
#pragma unroll
          for (int j = 0; j < NT; ++j) mma16816<INT8>(acc[t][j], a[0], a[1], a[2], a[3], b[j][0], b[j][1]);
        }
      }
    }
  };

  uint4 w0[4], w1[4], x0[NT], x1[NT];
  int k = kbeg + warp * kBatch;
  // halves that start past the slice are neither loaded nor multiplied
  if (k < kend) load_half(k, w0, x0);
  if (k + kHalf < kend) load_half(k + kHalf, w1, x1);
  int held = 0;
#pragma unroll 1
  for (int b = warp; b < nb; b += kRowsWarps) {
    const int kn = k + kRowsWarps * kBatch;
    multiply(w0, x0);
    if (kn < kend) load_half(kn, w0, x0);
    if (k + kHalf < kend) multiply(w1, x1);
    if (kn + kHalf < kend) load_half(kn + kHalf, w1, x1);
    k = kn;
    if constexpr (FINE) {
      const bool flush = ++held == kFlush;
      each([&](int t, int j, int e) {
        near[FINE ? t : 0][j][e] += acc[t][j][e];
        acc[t][j][e] = 0.f;
        if (flush) {
          far[FINE ? t : 0][j][e] += near[FINE ? t : 0][j][e];
          near[FINE ? t : 0][j][e] = 0.f;
        }
      });
      if (flush) held = 0;
    }
    if (INT8 && ++held == kFlush) {
      each([&](int t, int j, int e) {
        iacc[INT8 ? t : 0][j][e] += __float2int_rn(acc[t][j][e]);
        acc[t][j][e] = 0.f;
      });
      held = 0;
    }
  }

  if constexpr (FINE)
    each([&](int t, int j, int e) { acc[t][j][e] = near[FINE ? t : 0][j][e] + far[FINE ? t : 0][j][e]; });
  // accumulator element e of (tile t, group j): row of X, row of the strip
  const int words = R * kSumPitch;
  uint32_t *slot = red + warp * words;
  each([&](int t, int j, int e) {
    const int r = 8 * j + 2 * q + (e & 1), c = 16 * t + 8 * (e >> 1) + g;
    if (r < R)
      slot[r * kSumPitch + c] = INT8 ? (uint32_t)(iacc[INT8 ? t : 0][j][e] + __float2int_rn(acc[t][j][e]))
                                     : __float_as_uint(acc[t][j][e]);
  });
  __syncthreads();

  // the warps' sums in warp order, then the cluster's in rank order
  const int total = R * kStrip;
  const int64_t rows = p.NW - n0 < kStrip ? p.NW - n0 : kStrip;
  auto add = [](uint32_t a, uint32_t b) {
    return INT8 ? a + b : __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
  };
  auto block_sum = [&](int r, int c) {
    const uint32_t *s = red + r * kSumPitch + c;
    if (FINE) return add(add(s[0], s[words]), add(s[2 * words], s[3 * words]));
    uint32_t v = s[0];
#pragma unroll
    for (int i = 1; i < kRowsWarps; ++i) v = add(v, s[i * words]);
    return v;
  };
  if (p.cluster == 1) {
#pragma unroll 2
    for (int t = threadIdx.x; t < total; t += kRowsThreads) {
      const int r = t / kStrip, c = t % kStrip;
      if (c < rows) store_out(p, INT8, r * p.scr + (n0 + c) * p.scn, block_sum(r, c));
    }
    return;
  }
  uint32_t *part = red + kRowsWarps * words;
#pragma unroll 2
  for (int t = threadIdx.x; t < total; t += kRowsThreads) part[t] = block_sum(t / kStrip, t % kStrip);
  cluster_barrier();
  const uint32_t part_addr = smem_addr(part);
#pragma unroll 1
  for (int t = (int)rank * kRowsThreads + threadIdx.x; t < total; t += p.cluster * kRowsThreads) {
    const int r = t / kStrip, c = t % kStrip;
    uint32_t v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < p.cluster) v[j] = ld_cluster_u32(part_addr + 4u * t, j);
    uint32_t s = v[0];
#pragma unroll
    for (int j = 1; j < 8; ++j)
      if (j < p.cluster) s = add(s, v[j]);
    if (c < rows) store_out(p, INT8, r * p.scr + (n0 + c) * p.scn, s);
  }
  cluster_barrier();  // no block leaves while another may still read its sums
}

template <int NT, bool INT8, bool XVEC, bool FINE = false>
cudaError_t launch_nt(const RowsParams &p, int64_t strips, cudaStream_t st) {
  const size_t smem = (size_t)p.R * 4 * (kRowsWarps * kSumPitch + (p.cluster > 1 ? kStrip : 0));
  static_assert(8 * NT * 4 * (kRowsWarps * kSumPitch + kStrip) <= 48 * 1024, "no shared-memory opt-in needed");
  return launch_ex(gemm_rows_kernel<NT, INT8, XVEC, FINE>, dim3((unsigned)(strips * p.cluster)), dim3(kRowsThreads), smem,
                   st, p.cluster, p);
}

}  // namespace

// Strips, cluster size and K slice: the cluster (1-8 blocks along K) for
// which the rounds of resident blocks, each as long as its warps' batches
// plus the start and end of a block (about six batches), take least.  Clusters
// of four blocks and more do not fill every SM (a processing cluster's blocks are
// not a multiple of theirs): int8 4 x 2400 x 8192 in 75 clusters of 8 takes 9.9
// us, of 7 7.0, 4 x 2656 x 8192 in 83 of 7 11.2, of 6 7.2, 4 x 3200 x 8192 in 100
// of 6 11.5, of 5 8.1; 512 blocks do run at once.  bf16 against at most 8 rows
// has room for a fifth block per SM, which makes up for it (4 x 2400 x 8192 in 8
// 8.7, in 7 9.2).
int64_t rows_geometry(int64_t NW, int64_t K, int R, bool int8, int sms, int *cluster, int *kslice) {
  const int batch = int8 ? 128 : 64;
  const int64_t strips = (NW + kStrip - 1) / kStrip;
  const int64_t slots = (int64_t)kRowsBlocks * sms;
  const int64_t wide_slots = int8 || R > 8 ? slots * 22 / 25 : slots;
  double best = -1;
  for (int c = 1; c <= 8; ++c) {
    int64_t ks = (K + c - 1) / c;
    ks = (ks + batch - 1) / batch * batch;
    if (c > 1 && ks * (c - 1) >= K) continue;  // an empty slice
    const int64_t at_once = c >= 4 ? wide_slots : slots;
    const double cost = (double)((strips * c + at_once - 1) / at_once) * ((double)ks / (batch * kRowsWarps) + 6.0);
    if (best < 0 || cost < best) {
      best = cost;
      *cluster = c;
      *kslice = (int)ks;
    }
  }
  return strips;
}

// Whether the kernel is the fastest for these sizes.  A block streams its strip
// of W at what a few loads in flight give, about 3 us per 1024 k of bf16 and 1.8
// of int8, and a strip has at most eight blocks: with few strips a long K is
// faster on kernels that split it further: the CUDA-core kernel where it is the
// other choice (`few_m`: up to 2 rows of A for bf16 and 8 for int8), else the
// tensor cores.  Back to back, W stored N x K,
// this kernel / those: bf16 1 x 32 x 32768 8.5 / 18.7 us, x 65536 21.5 / 18.8; 1 x
// 128 x 16384 8.0 / 9.2, x 32768 15.1 / 10.5, x 131072 52.8 / 15.5; 1 x 600 x 8192
// 6.0 / 6.9, x 16384 9.4 / 8.7; 4 x 600 x 16384 9.2 / 10.1, x 32768 16.1 / 13.4;
// int8 1 x 32 x 65536 16.4 / 22.6; 1 x 128 x 32768 9.5 / 11.5, x 65536 16.6 / 12.1;
// 1 x 600 x 16384 6.6 / 7.4, x 32768 10.6 / 8.6.  From about 48 strips on the
// stream itself is the limit (1 x 2400 x 65536 bf16 50.0 / 60.2), but for long
// slices in more than one round (bf16 4 x 10000 x 16384 60.7 / 53.6).
bool rows_faster(int64_t NW, int64_t K, int R, bool int8, bool few_m, int sms) {
  int cluster, kslice;
  const int64_t strips = rows_geometry(NW, K, R, int8, sms, &cluster, &kslice), blocks = strips * cluster;
  if (strips * 16 >= (int64_t)sms * 5)  // 2.5 blocks per SM, were each strip given eight
    return int8 || R <= 2 || kslice <= 4096 || blocks <= (int64_t)kRowsBlocks * sms;
  if (int8) return !few_m || R > 8 || kslice <= (strips == 1 ? 8192 : strips <= 6 ? 4096 : 2560);
  if (!few_m || R > 2) return kslice <= 2560;
  return kslice <= (strips <= 2 ? 4096 : strips <= 6 ? 2048 : 1536);
}

cudaError_t launch_rows(const RowsParams &p, bool int8, int64_t strips, cudaStream_t st) {
  auto by_x = [&](auto nt, auto is_int8) {
    constexpr int NT = decltype(nt)::value;
    constexpr bool INT8 = decltype(is_int8)::value;
    return p.x_vec ? launch_nt<NT, INT8, true>(p, strips, st) : launch_nt<NT, INT8, false>(p, strips, st);
  };
  using std::integral_constant;
  if (!int8 && p.R <= 2)
    return p.x_vec ? launch_nt<1, false, true, true>(p, strips, st) : launch_nt<1, false, false, true>(p, strips, st);
  if (int8)
    return p.R > 8 ? by_x(integral_constant<int, 2>{}, std::true_type{}) : by_x(integral_constant<int, 1>{}, std::true_type{});
  return p.R > 8 ? by_x(integral_constant<int, 2>{}, std::false_type{}) : by_x(integral_constant<int, 1>{}, std::false_type{});
}

}  // namespace gb300
