// gemm_s8tm.cu -- exact int8 GEMM for shapes with a small operand: the large
// one is converted inside the kernel, straight into tensor memory.
//
// When one operand is much larger than the other (a batch of activations
// against a weight matrix, or a weight matrix a few columns wide), streaming
// and converting the large operand is most of the time.  The general int8
// path first stages both operands as bf16 (one launch that reads 1 byte and
// writes 2 per element), then the GEMM reads those 2 bytes again: 5 bytes of
// traffic per element of the large operand instead of 1.  This kernel stages
// only the small operand and streams the large one as int8:
//
//   P  the large operand, int8: B when M is small (P row = column n of C),
//      or A when N is small (P row = row m).  It is the MMA's 128-row A
//      operand, read from TMEM.  P is either K contiguous (A, or B stored
//      N x K) or P row contiguous (B stored K x N: the TMA box then holds
//      128 k-rows of 128 P rows, and the converters read it transposed).
//   Q  the small operand, staged beforehand (s8tm_stage_q_kernel) as the
//      exact shared-memory image the MMA reads for each (Q tile, k-block):
//      fp16, K-major, 128-byte swizzled, QN rows x 128 K = QN x 256 bytes,
//      contiguous; zero outside the matrix.  It is the MMA's QN-column B
//      operand.
//
// Roles (15 warps with QN = 64, 19 with QN = 128):
//   warp 0             P producer: per k-block of 128 a 128 x 128 int8 TMA
//                      box of P (128-byte rows, 128-byte swizzle) into a
//                      deep ring of its own.  Every row of a TMA box is a
//                      request of its own; 128-byte rows move twice the
//                      bytes per request of 64-byte ones (measured on
//                      GB300: twice the bytes per second per SM).
//   last warp          Q producer: Q's image with one bulk copy into a
//                      ring of its own (Q is read from L2).
//   8 converter warps  two groups of four that take alternate k-blocks:
//                      lane r of the warp with TMEM lane quadrant q converts
//                      P row 32 q + r (128 int8, read with eight
//                      conflict-free 16-byte loads) to 64 packed fp16 pairs
//                      and writes them to one of NA P slots in TMEM
//                      (tcgen05.st, lane = row, the lower k of a pair in the
//                      low half).  One group waits for its stores while the
//                      other converts; a single group left the MMAs idle for
//                      a store's latency per k-block (128 x 4096 x 4096 back
//                      to back 16.7 -> 12.9 us with the fp16 conversion,
//                      which takes half the instructions of the bf16 one).
//   warp 1             MMA issuer: tcgen05.mma kind::f16 with A in TMEM and
//                      B in shared memory, into one of two TMEM accumulators
//                      of QN fp32 columns.
//   4 or 8 warps       epilogue, 64 accumulator columns each: lane r of
//                      quadrant q owns P row 32 q + r.
//
// Exactness is the general int8 path's: every product is at most 2^14 in
// magnitude, so a partial sum of at most 1024 of them is an integer below
// 2^24 in magnitude and exact in fp32; the MMA warp closes the accumulator
// every 8 k-blocks of 128 (1024 K elements) and the epilogue converts each
// slab to int32 (exactly) and adds the slabs in int32 registers.
//
// A P stage is free again once every converter warp of its group has
// converted and stored its rows (one arrival per warp), a Q stage once the
// MMAs that read it have completed (tcgen05.commit), a TMEM P slot likewise.
// With P decoupled from the MMA, the P ring keeps its boxes in flight from
// HBM: measured on GB300, a P box takes about 2 us from issue to arrival
// under load.  What bounds a long unit is the k-block itself, 0.35 us for
// 128 x 128 x 128 (16 KB of P and 32 KB of Q from L2, and 0.27 us of MMA at its
// peak rate); short ones wait for their first box and their last slab.
#include <cuda_bf16.h>

#include "gemm_internal.h"

namespace gb300 {

namespace {

constexpr int kConvWarps = 4;   // converter warps of a group: one per TMEM lane quadrant
constexpr int kConvGroups = 2;  // groups, which take alternate k-blocks
constexpr int kEpiCols = 64;    // Q columns an epilogue thread accumulates
constexpr int kKB = kS8tmKB;                                      // K per k-block
constexpr uint32_t kPBytes = kBM * kKB;                           // 128 rows x 128 int8

// SP stages of P (16 KB each) and SQ of Q (QN x 256 bytes each) in two
// separate rings: a P stage is free again as soon as the converters have
// read it, so the P ring keeps SP boxes in flight from HBM whatever the MMA
// does; Q comes from L2 and needs only a few stages.
template <int QN, int SP, int SQ, int NA>
struct S8tmCfg {
  static_assert(QN == 64 || QN == 128, "QN is 64 or 128");
  // A converter group waits for a P stage by parity, so it may be at most one
  // phase ahead of the stage's use before: the same group's (an even ring), or
  // one whose MMA the group's free TMEM slot implies.
  static_assert(SP % kConvGroups == 0 && NA % kConvGroups == 0, "each stage and slot belongs to one group");
  static constexpr int kEpiWarps = 4 * (QN / kEpiCols);
  static constexpr int kQWarp = 2 + kEpiWarps + kConvGroups * kConvWarps;  // Q producer
  static constexpr int kThreads = (kQWarp + 1) * 32;
  static constexpr uint32_t kQHalf = QN * kRowBytes;  // QN x 64 fp16: one half of a Q image
  static constexpr uint32_t kQBytes = 2 * kQHalf;      // the k-block's Q image
  static constexpr uint32_t kPOffset = 0;
  static constexpr uint32_t kQOffset = SP * kPBytes;  // 1024-byte aligned
  // one 32 x 32 int32 block per epilogue warp, staging the TMA stores of C
  // (128-byte swizzle; 1024-byte aligned)
  static constexpr uint32_t kEpiOffset = kQOffset + SQ * kQBytes;
  static constexpr uint32_t kBarOffset = kEpiOffset + kEpiWarps * 4096;
  static constexpr uint32_t kNumBars = 2 * SP + 2 * SQ + 2 * NA + 5;
  static constexpr uint32_t kSmemBytes = kBarOffset + kNumBars * 8 + 16 + 1024;
  static_assert(kSmemBytes <= 232448, "shared memory per CTA is 227 KB");
  static constexpr uint32_t kPCol0 = 2 * QN;  // P slots (64 columns each) follow the two accumulators
  static constexpr uint32_t kTmemCols = pow2_at_least(2 * QN + 64 * NA);
  static_assert(kTmemCols <= 512, "TMEM has 512 columns");
};

struct S8tmUnit {
  int tp, tq, split, kb0, kb1;
};

__device__ __forceinline__ S8tmUnit decode_s8tm(const S8tmParams &p, int u) {
  const int tiles = p.tiles_p * p.tiles_q;
  S8tmUnit w;
  w.split = u / tiles;
  const int t = u - w.split * tiles;
  w.tp = t / p.tiles_q;  // the Q tiles of a P tile run side by side: P comes from HBM once
  w.tq = t - w.tp * p.tiles_q;
  w.kb0 = w.split * p.kb_per_split;
  w.kb1 = min(p.num_kb, w.kb0 + p.kb_per_split);
  return w;
}

// Stores the QN int32 sums of one P row: element i goes to offset
// off0 + i * step of the destination (C, or the split's partials), for the
// elements whose Q index q0 + i is inside the matrix; int32, or requantised
// to int16 / int8.  Where the elements are contiguous (C[prow][q]) a lane
// stores 16 bytes at a time: int16 8848 x 32 x 1648 unsplit 18.3 (general path)
// -> 13.0 us, int8 9616 x 64 x 3200 27.7 -> 15.0.  acc stays in registers.
template <int QN>
__device__ __forceinline__ void store_row(const S8tmParams &p, const int32_t (&acc)[QN], int split, int64_t off0,
                                          int64_t step, int64_t q0) {
  const int64_t nq = p.Q_rows - q0;  // valid elements (>= 1)
  if (p.add_into_c) {
    // int32 C, zeroed by the Q staging kernel: every split adds its exact
    // partial sums (integer addition, so any order gives the same C), here
    // element by element where C's alignment rules out TMA reductions
    int32_t *dst = reinterpret_cast<int32_t *>(p.C) + off0;
#pragma unroll
    for (int i = 0; i < QN; ++i)
      if (i < nq) atomicAdd(dst + i * step, acc[i]);
    return;
  }
  // Where the lane's elements are contiguous (C[prow][q]), 16 bytes at a time
  // with the widest stores their address allows.
  if (p.splits > 1 || p.out_bits == 32) {
    int32_t *dst = reinterpret_cast<int32_t *>(p.splits > 1 ? p.ws : p.C) +
                   (p.splits > 1 ? (int64_t)split * p.M * p.N : 0) + off0;
#pragma unroll
    for (int c = 0; c < QN; c += 4) {
      if (step == 1 && c + 4 <= nq) {
        const uint32_t w[4] = {(uint32_t)acc[c], (uint32_t)acc[c + 1], (uint32_t)acc[c + 2], (uint32_t)acc[c + 3]};
        store_chunk_aligned<4>(dst + c, w);
      } else {
#pragma unroll
        for (int i = c; i < c + 4; ++i)
          if (i < nq) dst[i * step] = acc[i];
      }
    }
    return;
  }
  const int32_t hi = (1 << (p.out_bits - 1)) - 1, lo = -hi - 1;
  const int esize = p.out_bits / 8;
  uint8_t *dst = reinterpret_cast<uint8_t *>(p.C) + off0 * esize;
  const bool words = step == 1 && (reinterpret_cast<uintptr_t>(dst) & 3) == 0;
#pragma unroll
  for (int c = 0; c < QN; c += 16) {
    uint32_t q[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) q[i] = (uint32_t)requantize_s32(acc[c + i], p.out_shift, lo, hi);
    if (words && c + 16 <= nq) {
      uint32_t h[4];
      if (esize == 2) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
#pragma unroll
          for (int i = 0; i < 4; ++i) h[i] = __byte_perm(q[8 * half + 2 * i], q[8 * half + 2 * i + 1], 0x5410);
          store_chunk_aligned<4>(dst + (c + 8 * half) * 2, h);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          h[i] = __byte_perm(__byte_perm(q[4 * i], q[4 * i + 1], 0x0040),
                             __byte_perm(q[4 * i + 2], q[4 * i + 3], 0x0040), 0x5410);
        store_chunk_aligned<4>(dst + c, h);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (c + i < nq) {
          if (esize == 2)
            reinterpret_cast<int16_t *>(dst)[(c + i) * step] = (int16_t)q[i];
          else
            reinterpret_cast<int8_t *>(dst)[(c + i) * step] = (int8_t)q[i];
        }
    }
  }
}

// int32 C by TMA: the warp's QN sums of its 32 P rows, 32 Q columns at a time,
// staged as a 32 x 32 block (128-byte rows, 16-byte chunk j of row r at chunk
// j ^ (r % 8)) and stored, or for split-K added into C by one TMA reduction
// (element-wise atomic); the TMA clips a block that crosses C's edges, and a
// block that starts outside C is not issued.  C[q][prow] (swap): block row =
// q, column = lane; else C[prow][q]: row = lane.
template <int QN>
__device__ __forceinline__ void out_rows_tma(bool add, const CUtensorMap *tm, uint32_t buf, int lane, const int32_t (&acc)[QN],
                                                bool swap, int32_t prow0, int32_t q0, int32_t P_rows, int32_t Q_rows) {
#pragma unroll
  for (int c = 0; c < QN / 32; ++c) {
    if (lane == 0) bulk_wait_read_all();  // the previous store has read the block
    __syncwarp();
    if (swap) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        st_shared_u32(buf + i * 128 + ((((uint32_t)lane >> 2) ^ ((uint32_t)i & 7u)) << 4) + ((uint32_t)lane & 3u) * 4,
                      static_cast<uint32_t>(acc[c * 32 + i]));
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        st_shared_v4(buf + lane * 128 + (((uint32_t)j ^ ((uint32_t)lane & 7u)) << 4),
                     static_cast<uint32_t>(acc[c * 32 + 4 * j]), static_cast<uint32_t>(acc[c * 32 + 4 * j + 1]),
                     static_cast<uint32_t>(acc[c * 32 + 4 * j + 2]), static_cast<uint32_t>(acc[c * 32 + 4 * j + 3]));
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0 && prow0 < P_rows && q0 + c * 32 < Q_rows) {
      const int32_t x = swap ? prow0 : q0 + c * 32, y = swap ? q0 + c * 32 : prow0;
      if (add)
        tma_reduce_add_2d(tm, buf, x, y);
      else
        tma_store_2d(tm, buf, x, y);
      bulk_commit();
    }
  }
}

template <int QN, int SP, int SQ, int NA, bool PK>
__global__ void __launch_bounds__(S8tmCfg<QN, SP, SQ, NA>::kThreads, 1)
    gemm_s8tm_kernel(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmC,
                     const S8tmParams p) {
  using Cfg = S8tmCfg<QN, SP, SQ, NA>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // swizzle atoms need 1024-byte alignment
  uint8_t *base_ptr = smem_raw + (base - raw);
  const uint32_t sP = base + Cfg::kPOffset;
  const uint32_t sQ = base + Cfg::kQOffset;
  const uint32_t bars = base + Cfg::kBarOffset;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(base_ptr + Cfg::kBarOffset + Cfg::kNumBars * 8);
  volatile uint32_t *abort_flag = tmem_slot + 1;

  // P ring, Q ring, TMEM P slots, accumulators
  auto pfull_bar = [&](uint32_t s) { return bars + 8u * s; };
  auto pempty_bar = [&](uint32_t s) { return bars + 8u * (SP + s); };
  auto qfull_bar = [&](uint32_t s) { return bars + 8u * (2 * SP + s); };
  auto qempty_bar = [&](uint32_t s) { return bars + 8u * (2 * SP + SQ + s); };
  auto tfull_bar = [&](uint32_t a) { return bars + 8u * (2 * SP + 2 * SQ + a); };
  auto tempty_bar = [&](uint32_t a) { return bars + 8u * (2 * SP + 2 * SQ + NA + a); };
  auto accf_bar = [&](uint32_t b) { return bars + 8u * (2 * SP + 2 * SQ + 2 * NA + b); };
  auto acce_bar = [&](uint32_t b) { return bars + 8u * (2 * SP + 2 * SQ + 2 * NA + 2 + b); };
  const uint32_t drain_bar = bars + 8u * (2 * SP + 2 * SQ + 2 * NA + 4);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // warp-uniform for the compiler
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SP; ++s) {
      mbar_init(pfull_bar(s), 1);
      mbar_init(pempty_bar(s), kConvWarps);
    }
    for (int s = 0; s < SQ; ++s) {
      mbar_init(qfull_bar(s), 1);
      mbar_init(qempty_bar(s), 1);
    }
    for (int a = 0; a < NA; ++a) {
      mbar_init(tfull_bar(a), kConvWarps);
      mbar_init(tempty_bar(a), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf_bar(b), 1);
      mbar_init(acce_bar(b), Cfg::kEpiWarps * 32);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0u;
    fence_mbar_init();
    tma_prefetch_desc(&tmP);
    if (p.c_tma) tma_prefetch_desc(&tmC);
  }
  if (warp == 1) tmem_alloc<Cfg::kTmemCols>(smem_addr(tmem_slot));
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // The previous kernel of the stream is the Q staging launch.  This one
  // starts after everything before that launch has completed: it is either a
  // plain launch, or a programmatic one that lets this grid start only when
  // it ends.  It writes Q's images and, for split-K into int32 C, zeroes C:
  // the Q producer and the epilogue wait for it (griddep_wait) before touching
  // those, while P, written before, is streamed at once.

  const int num_units = p.tiles_p * p.tiles_q * p.splits;
  constexpr uint64_t kDrainNs = 200ull * 1000 * 1000;

  if (warp == 0 || warp == Cfg::kQWarp) {
    // -------------------------------------------- producers (P, then Q)
    const bool is_p = warp == 0;
    if (!is_p) griddep_wait();
    const uint32_t ns = is_p ? SP : SQ;
    uint32_t s = 0, ph = 0, g = 0;  // stage, its phase, copies issued
    bool ok = true;
    for (int u = blockIdx.x; ok && u < num_units; u += gridDim.x) {
      const S8tmUnit w = decode_s8tm(p, u);
      const uint8_t *q_src = static_cast<const uint8_t *>(p.q_img) + (int64_t)w.tq * p.num_kb * (int64_t)Cfg::kQBytes;
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        if (!mbar_wait_warp(is_p ? pempty_bar(s) : qempty_bar(s), ph ^ 1u, abort_flag, p.err, p.wait_limit_ns)) {
          ok = false;
          break;
        }
        if (elect_one()) {
          if (is_p) {
            mbar_arrive_expect_tx(pfull_bar(s), kPBytes);
            if constexpr (PK)
              tma_load_2d(sP + s * kPBytes, &tmP, kb * kKB, w.tp * kBM, pfull_bar(s));
            else
              tma_load_2d(sP + s * kPBytes, &tmP, w.tp * kBM, kb * kKB, pfull_bar(s));
          } else {
            mbar_arrive_expect_tx(qfull_bar(s), Cfg::kQBytes);
            bulk_load(sQ + s * Cfg::kQBytes, q_src + (int64_t)kb * (int64_t)Cfg::kQBytes, Cfg::kQBytes, qfull_bar(s));
          }
        }
        __syncwarp();
        ++g;
        if (++s == ns) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    // Every copy this warp issued has landed before the CTA may exit.
    const uint32_t first = g > ns ? g - ns : 0u;
    for (uint32_t i = first; i < g; ++i)
      mbar_wait_drain(is_p ? pfull_bar(i % ns) : qfull_bar(i % ns), (i / ns) & 1u, kDrainNs);
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA issuer
    constexpr uint32_t idesc = idesc_f16_f32(kBM, QN);
    // K-major, 128-byte swizzle, 8-row atoms 1024 bytes apart
    const uint64_t dq = smem_desc_sw128(sQ, 16, 1024);
    uint32_t s = 0, ph = 0, a = 0, tph = 0, acc_cnt = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < num_units; u += gridDim.x) {
      const S8tmUnit w = decode_s8tm(p, u);
      for (int kb_s = w.kb0; ok && kb_s < w.kb1; kb_s += p.slab_kb) {
        const int kb_e = min(w.kb1, kb_s + p.slab_kb);
        const uint32_t b = acc_cnt & 1u, aph = (acc_cnt >> 1) & 1u;
        if (!mbar_wait_warp(acce_bar(b), aph ^ 1u, abort_flag, p.err, p.wait_limit_ns)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + b * QN;
        for (int kb = kb_s; kb < kb_e; ++kb) {
          if (!mbar_wait_warp(qfull_bar(s), ph, abort_flag, p.err, p.wait_limit_ns) ||
              !mbar_wait_warp(tfull_bar(a), tph, abort_flag, p.err, p.wait_limit_ns)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          if (elect_one()) {
            const uint64_t q0 = dq + s * (Cfg::kQBytes / 16);
            const uint32_t a_tmem = tmem_base + Cfg::kPCol0 + a * 64;
#pragma unroll
            for (int k = 0; k < kKB / 16; ++k)
              // one K step of 16 is 8 packed columns of the P slot, and 32
              // bytes along the rows of Q's half k / 4
              tc_mma_f16_tmem_a(d_tmem, a_tmem + k * 8, q0 + (k >> 2) * (Cfg::kQHalf / 16) + (k & 3) * 2, idesc,
                                 (kb > kb_s || k > 0) ? 1u : 0u);
            tc_commit(qempty_bar(s));  // the Q stage may be refilled once these MMAs finish
            tc_commit(tempty_bar(a));  // and the P slot reused
          }
          __syncwarp();
          if (++s == SQ) {
            s = 0;
            ph ^= 1u;
          }
          if (++a == NA) {
            a = 0;
            tph ^= 1u;
          }
        }
        if (!ok) break;
        if (elect_one()) tc_commit(accf_bar(b));
        __syncwarp();
        ++acc_cnt;
      }
    }
    if (elect_one()) tc_commit(drain_bar);
    __syncwarp();
    mbar_wait_drain(drain_bar, 0, kDrainNs);
    __syncwarp();
  } else if (warp >= 2 + Cfg::kEpiWarps) {
    // ------------------------------------------------------- converters
    // Two groups of four warps take alternate k-blocks: while one waits for
    // its TMEM stores and publishes its slot, the other converts.
    const int quad = warp & 3;
    const int r = quad * 32 + lane;               // P row within the tile = TMEM lane
    const uint32_t sw = (uint32_t)r & 7u;         // 128-byte swizzle: chunk j at j ^ (r % 8)
    const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + Cfg::kPCol0;
    const uint32_t group = (uint32_t)(warp - 2 - Cfg::kEpiWarps) / kConvWarps;
    uint32_t g = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < num_units; u += gridDim.x) {
      const S8tmUnit w = decode_s8tm(p, u);
      for (int kb = w.kb0; kb < w.kb1; ++kb, ++g) {
        if ((g & (kConvGroups - 1)) != group) continue;
        const uint32_t s = g % SP, ph = (g / SP) & 1u;
        const uint32_t a = g % NA, tph = (g / NA) & 1u;
        if (!mbar_wait_warp(pfull_bar(s), ph, abort_flag, p.err, p.wait_limit_ns) ||
            !mbar_wait_warp(tempty_bar(a), tph ^ 1u, abort_flag, p.err, p.wait_limit_ns)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        uint32_t o[64];  // o[c]: fp16 of k = 2c (low half) and 2c + 1
        if constexpr (PK) {
          const uint32_t row = sP + s * kPBytes + (uint32_t)r * kKB;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 v = ld_shared_v4(row + (((uint32_t)j ^ sw) << 4));  // k = 16 j .. 16 j + 15
            s8x4_to_f16x4(v.x, o[8 * j + 0], o[8 * j + 1]);
            s8x4_to_f16x4(v.y, o[8 * j + 2], o[8 * j + 3]);
            s8x4_to_f16x4(v.z, o[8 * j + 4], o[8 * j + 5]);
            s8x4_to_f16x4(v.w, o[8 * j + 6], o[8 * j + 7]);
          }
        } else {
          // The box holds 128 k-rows of 128 P rows (byte r of k-row k in
          // chunk (r / 16) ^ (k % 8)).  Lane r reads the 32-bit word holding
          // its byte from four consecutive k-rows (lanes r, r ^ 1, r ^ 2,
          // r ^ 3 read the same word; the warp's 32 rows span two chunks, so
          // the reads are conflict-free) and gathers byte r % 4 of each into
          // one word of four consecutive k.
          const uint32_t box = sP + s * kPBytes;
          const uint32_t rc = (uint32_t)r >> 4, rw = (uint32_t)r & 12u;
          const uint32_t sel = ((uint32_t)r & 3u) | ((4u + ((uint32_t)r & 3u)) << 4);
#pragma unroll
          for (int kq = 0; kq < kKB / 4; ++kq) {
            uint32_t w4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint32_t k = 4u * kq + i;
              w4[i] = ld_shared_u32(box + k * 128u + ((rc ^ (k & 7u)) << 4) + rw);
            }
            const uint32_t x = __byte_perm(__byte_perm(w4[0], w4[1], sel), __byte_perm(w4[2], w4[3], sel), 0x5410);
            s8x4_to_f16x4(x, o[2 * kq], o[2 * kq + 1]);
          }
        }
        tmem_st_32x32b_x64(lane_base + a * 64, o);
        __syncwarp();
        // The P stage is released only after that store was issued, which
        // needed every byte this warp reads of it.  An arrival right after the
        // shared-memory loads were issued let the refill overtake them while
        // the load queue was backed up (single 16-byte pieces of P wrong).
        if (lane == 0) mbar_arrive(pempty_bar(s));
        __syncwarp();
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(tfull_bar(a));  // hand the slot to the MMA warp
        __syncwarp();
      }
    }
  } else {
    // --------------------------------------------------------- epilogue
    griddep_wait();  // C (zeroed by the staging launch) is written below
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    const int col0 = ((warp - 2) >> 2) * kEpiCols;  // this warp's Q columns of the tile
    uint32_t acc_cnt = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < num_units; u += gridDim.x) {
      const S8tmUnit w = decode_s8tm(p, u);
      int32_t acc[kEpiCols];
#pragma unroll
      for (int i = 0; i < kEpiCols; ++i) acc[i] = 0;
      for (int kb_s = w.kb0; kb_s < w.kb1; kb_s += p.slab_kb) {
        const uint32_t b = acc_cnt & 1u, aph = (acc_cnt >> 1) & 1u;
        if (!mbar_wait_warp(accf_bar(b), aph, abort_flag, p.err, p.wait_limit_ns)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t t0 = tmem_base + b * QN + ((uint32_t)(quad * 32) << 16) + col0;
#pragma unroll
        for (int c = 0; c < kEpiCols / 16; ++c) {
          uint32_t v[16];
          tmem_ld_32x32b_x16(t0 + c * 16, v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[c * 16 + i] += __float2int_rn(__uint_as_float(v[i]));
        }
        tc_fence_before_sync();
        mbar_arrive(acce_bar(b));
        ++acc_cnt;
      }
      if (!ok) break;
      const int64_t q0 = (int64_t)w.tq * QN + col0;
      if (q0 >= p.Q_rows) continue;
      if (p.c_tma) {  // the whole warp: rows past the matrix are clipped by the TMA
        out_rows_tma<kEpiCols>(p.add_into_c != 0, &tmC, base + Cfg::kEpiOffset + (warp - 2) * 4096, lane, acc, p.swap != 0,
                                  w.tp * kBM + quad * 32, (int32_t)q0, p.P_rows, p.Q_rows);
        continue;
      }
      const int64_t prow = (int64_t)w.tp * kBM + r;
      if (prow >= p.P_rows) continue;
      // partials (split-K of int16 / int8 outputs) have row pitch N; C has ldc
      const int64_t ld = (p.splits > 1 && p.out_bits != 32) ? (int64_t)p.N : p.ldc;
      if (p.swap)  // C[q][prow]: per element the warp's lanes store 32 consecutive columns
        store_row<kEpiCols>(p, acc, w.split, q0 * ld + prow, ld, q0);
      else         // C[prow][q]
        store_row<kEpiCols>(p, acc, w.split, prow * ld + q0, 1, q0);
    }
  }

  // the epilogue's TMA stores have completed before the CTA leaves
  if (p.c_tma && warp >= 2 && warp < 2 + Cfg::kEpiWarps && lane == 0) bulk_wait_all();
  griddep_launch_dependents();  // e.g. the split-K reduction may start setting up
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after_sync();
    tmem_dealloc<Cfg::kTmemCols>(tmem_base);
  }
}

// Q's image for one (Q tile, k-block): QN rows x 128 K of fp16 as two
// 64-K halves of QN 128-byte rows, 16-byte chunk j of row r stored at chunk
// j ^ (r % 8) (the 128-byte swizzle).  One thread writes one 16-byte chunk
// (8 consecutive k of one row), reading Q(q, k) at src + q * sq + k * sk.
__global__ void __launch_bounds__(256)
    s8tm_stage_q_kernel(const int8_t *__restrict__ src, int64_t sq, int64_t sk, int Q_rows, int K, int qn,
                        int num_kb, uint4 *__restrict__ img, int64_t chunks, int32_t *__restrict__ zero_c,
                        int64_t c_rows, int64_t c_cols, int64_t ldc, int overlap) {
  if (overlap) griddep_launch_dependents();  // the GEMM streams P now and waits for completion before reading Q
  griddep_wait();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= chunks) {  // the remaining threads zero C (int32, the splits' sums are added into it)
    if (!zero_c) return;
    // four consecutive elements of a row per step, with one 16-byte store
    // when the row pitch and base allow it
    const bool vec = (reinterpret_cast<uintptr_t>(zero_c) & 15) == 0 && (ldc & 3) == 0;
    const int64_t quads = (c_cols + 3) >> 2, total = c_rows * quads;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x - chunks;
    for (int64_t e = t - chunks; e < total; e += stride) {
      const int64_t r = e / quads, c = (e - r * quads) << 2;
      int32_t *dst = zero_c + r * ldc + c;
      if (vec && c + 4 <= c_cols) {
        *reinterpret_cast<int4 *>(dst) = make_int4(0, 0, 0, 0);
      } else {
        for (int i = 0; i < 4 && c + i < c_cols; ++i) dst[i] = 0;
      }
    }
    return;
  }
  const int per_tile = 2 * qn * 8;  // 16-byte chunks per image
  const int64_t tile = t / per_tile;
  const int c = (int)(t - tile * per_tile);
  const int h = c / (qn * 8), rem = c - h * (qn * 8);
  const int row = rem >> 3, j = rem & 7;
  const int64_t tq = tile / num_kb, kb = tile - tq * num_kb;
  const int64_t q = tq * qn + row, k0 = kb * kKB + h * 64 + j * 8;
  uint32_t w[2] = {0u, 0u};
  if (q < Q_rows) {
    const int8_t *s = src + q * sq + k0 * sk;
    if (sk == 1 && k0 + 8 <= K && (reinterpret_cast<uintptr_t>(s) & 7) == 0) {
      const uint2 v = *reinterpret_cast<const uint2 *>(s);
      w[0] = v.x;
      w[1] = v.y;
    } else {
      for (int i = 0; i < 8; ++i)
        if (k0 + i < K) w[i >> 2] |= (uint32_t)(uint8_t)s[i * sk] << (8 * (i & 3));
    }
  }
  uint4 o;
  s8x4_to_f16x4(w[0], o.x, o.y);
  s8x4_to_f16x4(w[1], o.z, o.w);
  const int64_t at = tile * per_tile + h * (qn * 8) + row * 8 + (j ^ (row & 7));
  img[at] = o;
}

template <int QN, int SP, int SQ, int NA, bool PK>
cudaError_t launch_one(const CUtensorMap &tp, const CUtensorMap &tc, const S8tmParams &p, int grid,
                       cudaStream_t st) {
  using Cfg = S8tmCfg<QN, SP, SQ, NA>;
  auto kern = gemm_s8tm_kernel<QN, SP, SQ, NA, PK>;
  // the shared-memory opt-in is per device and kernel: set it once
  static bool opted_in[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !opted_in[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmemBytes);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) opted_in[dev] = true;
  }
  return launch_ex(kern, dim3(grid), dim3(Cfg::kThreads), Cfg::kSmemBytes, st, 1, tp, tc, p);
}

}  // namespace

size_t s8tm_q_image_bytes(int qn, int64_t Q_rows, int64_t K) {
  const int64_t tiles_q = (Q_rows + qn - 1) / qn, num_kb = (K + kKB - 1) / kKB;
  return (size_t)tiles_q * num_kb * 2 * qn * 128;
}

cudaError_t launch_s8tm_stage_q(const int8_t *src, int64_t sq, int64_t sk, int64_t Q_rows, int64_t K, int qn,
                                void *img, int32_t *zero_c, int64_t c_rows, int64_t c_cols, int64_t ldc,
                                int64_t p_bytes, cudaStream_t st) {
  // A plain launch, after which everything earlier on the stream has
  // completed, lets the GEMM stream P while Q is staged; a programmatic one is
  // scheduled while the previous kernel drains, but the GEMM then starts when
  // it ends.  Measured on GB300, calls back to back (plain / programmatic):
  // 64 x 2048 x 2048 8.2 / 7.1 us, 32 x 4096 x 4096 12.3 / 10.9, 128 x 4096 x
  // 4096 14.3 / 12.9, 128 x 12288 x 4096 20.6 / 22.0, 8192 x 64 x 8192 20.8 /
  // 21.3.  Replayed from a graph the plain one is faster at every size (128 x 4096
  // x 4096 12.8 / 14.1, 64 x 2048 x 2048 7.0 / 7.2).
  constexpr int64_t kStageOverlapBytes = int64_t(32) << 20;
  const int64_t num_kb = (K + kKB - 1) / kKB;
  const int64_t chunks = (int64_t)s8tm_q_image_bytes(qn, Q_rows, K) / 16;
  // more threads zero C when asked (up to 64K, a grid-stride loop over
  // four-element pieces of its rows)
  const int64_t quads = zero_c ? c_rows * ((c_cols + 3) / 4) : 0;
  const int64_t extra = quads < 65536 ? quads : 65536;
  if (chunks + extra == 0) return cudaSuccess;
  const dim3 grid((unsigned)((chunks + extra + 255) / 256));
  if (p_bytes >= kStageOverlapBytes || !pdl_enabled() || capturing(st)) {
    s8tm_stage_q_kernel<<<grid, 256, 0, st>>>(src, sq, sk, (int)Q_rows, (int)K, qn, (int)num_kb,
                                              static_cast<uint4 *>(img), chunks, zero_c, c_rows, c_cols, ldc, 1);
    return cudaGetLastError();
  }
  return launch_ex(s8tm_stage_q_kernel, grid, dim3(256), 0, st, 1, src, sq, sk, (int)Q_rows, (int)K, qn, (int)num_kb,
                   static_cast<uint4 *>(img), chunks, zero_c, c_rows, c_cols, ldc, 0);
}

cudaError_t launch_s8tm(int qn, bool p_kmajor, const CUtensorMap &tp, const CUtensorMap &tc, const S8tmParams &p,
                        int grid, cudaStream_t st) {
  // P stages x 16 KB + Q stages x (QN x 256 bytes) + a 4 KB block per
  // epilogue warp: 6 x 16 + 3 x 32 + 32 KB (QN 128) or 8 x 16 + 5 x 16 +
  // 16 KB (QN 64); TMEM: two accumulators and four (six) 64-column P slots.
  // Q, read from L2 by every CTA, is up to twice P's bytes: with two Q stages
  // its latency set the pace (128 x 4096 x 11008 19.3 us, with three 17.2).
  if (qn == 128)
    return p_kmajor ? launch_one<128, 6, 3, 4, true>(tp, tc, p, grid, st)
                    : launch_one<128, 6, 3, 4, false>(tp, tc, p, grid, st);
  return p_kmajor ? launch_one<64, 8, 5, 6, true>(tp, tc, p, grid, st)
                  : launch_one<64, 8, 5, 6, false>(tp, tc, p, grid, st);
}

}  // namespace gb300
