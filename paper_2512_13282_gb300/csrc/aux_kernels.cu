// aux_kernels.cu -- the memory-bound helpers around the tensor-core kernel:
// operand staging (int8 -> bf16, re-pitching misaligned bf16), zero fill for
// K == 0, and the split-K reduction (with the int8 path's requantisation).
#include <cuda_bf16.h>

#include <cstring>

#include "gemm_internal.h"

namespace gb300 {

namespace {

constexpr int kThreads = 256;

inline int grid_for(int64_t work, int per_thread, int sms) {
  const int64_t want = (work + (int64_t)kThreads * per_thread - 1) / ((int64_t)kThreads * per_thread);
  const int64_t cap = (int64_t)sms * 8;
  return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

// int8 -> bf16 bit pattern.  |v| <= 128 needs 8 significant bits, which a
// bf16 has, so the float's upper half is the exact bf16 (low half is zero).
__device__ __forceinline__ uint32_t s8_to_bf16_bits(int v) {
  return __float_as_uint(static_cast<float>(v)) >> 16;
}

// Converts 16 int8 held in a uint4 to 16 bf16 bit patterns in two uint4.
__device__ __forceinline__ void s8x16_to_bf16x16(const int4 raw, uint4 &lo, uint4 &hi) {
  uint32_t o[8];
  s8x4_to_bf16x4((uint32_t)raw.x, o[0], o[1]);
  s8x4_to_bf16x4((uint32_t)raw.y, o[2], o[3]);
  s8x4_to_bf16x4((uint32_t)raw.z, o[4], o[5]);
  s8x4_to_bf16x4((uint32_t)raw.w, o[6], o[7]);
  lo = make_uint4(o[0], o[1], o[2], o[3]);
  hi = make_uint4(o[4], o[5], o[6], o[7]);
}

constexpr int kS8Threads = 256;

// Row piece -> (row, first column) for pieces of `w` elements, `cpr` pieces
// per row (32-bit division where the index allows it).
__device__ __forceinline__ void piece_rc(uint64_t u, uint32_t cpr, int w, int64_t &r, int64_t &c) {
  uint64_t rr, q;
  if (u <= 0xFFFFFFFFull) {
    rr = (uint32_t)u / cpr;
    q = (uint32_t)u - (uint32_t)rr * cpr;
  } else {
    rr = u / cpr;
    q = u - rr * cpr;
  }
  r = (int64_t)rr;
  c = (int64_t)q * w;
}

// The staging and re-pitch kernels are programmatic launches that wait for the
// previous kernel at their start: a plain launch in the chain of a stream's
// kernels costs up to 2 us more on GB300 (int8 1024^3 back to back 10.3 -> 9.8
// us).  Replayed from a graph it is the other way round (1376 x 3276 x 112 10.9
// us programmatic, 8.6 plain; 2048^3 23.1 and 22.0), so that captured launches are
// plain.  Either way everything before them has completed when they let the next
// kernel start, which sets itself up while they run and shares the GPU with them
// alone.
__device__ __forceinline__ void staging_begins() {
  griddep_wait();
  griddep_launch_dependents();
}
template <typename... KArgs, typename... Args>
cudaError_t launch_staging(void (*kern)(KArgs...), int64_t threads, cudaStream_t st, Args... args) {
  const dim3 grid((unsigned)((threads + kS8Threads - 1) / kS8Threads));
  if (!capturing(st)) return launch_ex(kern, grid, dim3(kS8Threads), 0, st, 1, args...);
  kern<<<grid, kS8Threads, 0, st>>>(args...);
  return cudaGetLastError();
}

// General path (any alignment, any leading dimension): both matrices as one
// flat list of 16-element row pieces -- piece t < items_a is piece t % cpr_a
// of row t / cpr_a of A (cpr = pieces per row), the rest likewise of B.  A
// thread reads its 16 bytes with the widest loads the row's address allows
// (odd rows as five aligned words, shifted; byte by byte they took 1.5 times
// the GEMM's own time at 1001 x 1503 x 3001) and writes 32 bytes with two
// 16-byte stores (staged rows start 16-byte aligned).  A row's last, partial
// piece does the same where its 16 bytes lie inside the matrix and its 32 inside
// the staged row: what follows the row is read, converted and never used (element
// by element, each load waited for, they set the time of short rows).
__global__ void __launch_bounds__(kS8Threads)
    s8_to_bf16_pair_kernel(const S8Job a, const S8Job b, uint32_t cpr_a, uint32_t cpr_b, uint64_t items_a,
                           uint64_t items) {
  staging_begins();
  const uint64_t t = (uint64_t)blockIdx.x * kS8Threads + threadIdx.x;
  if (t >= items) return;
  const bool in_a = t < items_a;
  const S8Job &j = in_a ? a : b;
  int64_t r, c;
  piece_rc(in_a ? t : t - items_a, in_a ? cpr_a : cpr_b, 16, r, c);
  const int8_t *src = j.src + r * j.ld_src + c;
  uint16_t *dst = j.dst + r * j.ld_dst + c;
  const uint8_t *lo8 = reinterpret_cast<const uint8_t *>(j.src), *hi8 = lo8 + (j.rows - 1) * j.ld_src + j.cols;
  if (c + 16 <= j.cols || (c + 16 <= j.ld_dst && reinterpret_cast<const uint8_t *>(src) + 16 <= hi8)) {
    const uint4 v = load16_any<true>(reinterpret_cast<const uint8_t *>(src), lo8, hi8);
    const int4 raw = make_int4((int)v.x, (int)v.y, (int)v.z, (int)v.w);
    uint4 lo, hi;
    s8x16_to_bf16x16(raw, lo, hi);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    d[0] = lo;
    d[1] = hi;
  } else {
    for (int64_t i = 0; c + i < j.cols; ++i) dst[i] = (uint16_t)s8_to_bf16_bits(src[i]);
  }
}

// Dense fast path: both matrices contiguous (leading dimension = columns,
// source 16-byte aligned), so each is one flat array; thread v converts
// 16-element vector v (v < va: of A, else of B) with one 16-byte load and
// two 16-byte stores, over a grid that covers every vector once (measured on
// GB300 faster than fewer threads looping over several vectors).  A last
// partial vector (elements % 16) is converted element by element.
__global__ void __launch_bounds__(kS8Threads)
    s8_to_bf16_dense_kernel(const S8Job a, const S8Job b, int64_t na, int64_t nb) {
  staging_begins();
  const int64_t va = (na + 15) / 16, vtot = va + (nb + 15) / 16;
  const int64_t v = (int64_t)blockIdx.x * kS8Threads + threadIdx.x;
  if (v >= vtot) return;
  const bool in_a = v < va;
  const S8Job &j = in_a ? a : b;
  const int64_t n = in_a ? na : nb;
  const int64_t e = (in_a ? v : v - va) * 16;
  if (e + 16 <= n) {
    const int4 raw = __ldcs(reinterpret_cast<const int4 *>(j.src + e));
    uint4 lo, hi;
    s8x16_to_bf16x16(raw, lo, hi);
    uint4 *d = reinterpret_cast<uint4 *>(j.dst + e);
    d[0] = lo;
    d[1] = hi;
  } else {
    for (int64_t i = e; i < n; ++i) j.dst[i] = (uint16_t)s8_to_bf16_bits(j.src[i]);
  }
}

// Re-pitch of a bf16 matrix into a buffer whose rows start 16-byte aligned:
// thread t copies 8-element piece t % cpr of row t / cpr with one 16-byte
// store (the source and a row's last piece as for the int8 staging above).
__global__ void __launch_bounds__(kS8Threads)
    pack_u16_kernel(const uint16_t *__restrict__ src, int64_t rows, int64_t cols, int64_t ld_src,
                    uint16_t *__restrict__ dst, int64_t ld_dst, uint32_t cpr, uint64_t items) {
  staging_begins();
  const uint64_t t = (uint64_t)blockIdx.x * kS8Threads + threadIdx.x;
  if (t >= items) return;
  int64_t r, c;
  piece_rc(t, cpr, 8, r, c);
  const uint16_t *s = src + r * ld_src + c;
  uint16_t *d = dst + r * ld_dst + c;
  const uint8_t *lo = reinterpret_cast<const uint8_t *>(src), *hi = lo + ((rows - 1) * ld_src + cols) * 2;
  if (c + 8 <= cols || reinterpret_cast<const uint8_t *>(s) + 16 <= hi) {
    *reinterpret_cast<uint4 *>(d) = load16_any<true>(reinterpret_cast<const uint8_t *>(s), lo, hi);
  } else {
    for (int64_t i = 0; c + i < cols; ++i) d[i] = s[i];
  }
}

template <typename T>
__global__ void zero_fill_kernel(T *C, int64_t M, int64_t N, int64_t ldc) {
  const int64_t total = M * N;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / N, c = t - r * N;
    C[r * ldc + c] = T(0);
  }
}

// Split-K reduction: thread t sums 4-element piece t % cpr of row t / cpr
// over the splits in a fixed order (split 0, 1, ...), with 16-byte partial
// loads when N is a multiple of 4, and stores the piece with one store where
// C's address allows it.
struct Piece {
  int64_t r, c;
  int n;      // elements in the piece (4, or fewer at the end of a row)
  int64_t w;  // offset of its first element in a plane of partials
};

__device__ __forceinline__ Piece piece_of(uint64_t t, uint32_t cpr, int64_t N) {
  uint64_t r, q;
  if (t <= 0xFFFFFFFFull) {
    r = (uint32_t)t / cpr;
    q = (uint32_t)t - (uint32_t)r * cpr;
  } else {
    r = t / cpr;
    q = t - r * cpr;
  }
  Piece pc;
  pc.r = (int64_t)r;
  pc.c = (int64_t)q * 4;
  pc.n = N - pc.c < 4 ? (int)(N - pc.c) : 4;
  pc.w = pc.r * N + pc.c;
  return pc;
}

// Piece t of the part of C that rt covers; false when it lies outside C.
// Partials of all of C are planes of C's shape; those of a split tail are
// compact: per plane, tile i of the tail as rows x cols words at row
// i * rows.
__device__ __forceinline__ bool reduce_piece(uint64_t t, uint32_t cpr, int64_t M, int64_t N, const ReduceTiles &rt,
                                             Piece *pc) {
  if (rt.count == 0) {
    if (t >= (uint64_t)M * cpr) return false;
    *pc = piece_of(t, cpr, N);
    return true;
  }
  const uint32_t cpt = (uint32_t)rt.cols / 4;
  const uint64_t per_tile = (uint64_t)rt.rows * cpt;
  if (t >= per_tile * (uint64_t)rt.count) return false;
  const int ti = (int)(t / per_tile);
  const uint32_t rem = (uint32_t)(t - (uint64_t)ti * per_tile);
  int tm, tn;
  raster_tile(rt.first + ti, rt.tiles_m, rt.tiles_n, rt.group_m, &tm, &tn);
  const uint32_t rl = rem / cpt, cl = (rem % cpt) * 4;
  pc->r = (int64_t)tm * rt.rows + rl;
  pc->c = (int64_t)tn * rt.cols + cl;
  if (pc->r >= M || pc->c >= N) return false;
  pc->n = N - pc->c < 4 ? (int)(N - pc->c) : 4;
  pc->w = ((int64_t)ti * rt.rows + rl) * rt.cols + cl;
  return true;
}

// Sum of a piece over the planes (plane stride MN words); vec: the
// pieces of a plane start on 16-byte boundaries.
template <typename T>
__device__ __forceinline__ void sum_piece(const T *__restrict__ ws, int splits, int64_t MN, bool vec,
                                          const Piece &pc, T (&v)[4]) {
  const int64_t base = pc.w;
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = T(0);
  if (pc.n == 4 && vec) {
    // the planes in order, four loads in flight at a time (one after the
    // other would cost a memory latency per plane)
    for (int k = 0; k < splits; k += 4) {
      uint4 w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (k + j < splits) w[j] = __ldcs(reinterpret_cast<const uint4 *>(ws + (int64_t)(k + j) * MN + base));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (k + j >= splits) break;
        T x[4];
        memcpy(x, &w[j], sizeof w[j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] += x[i];
      }
    }
  } else {
    for (int k = 0; k < splits; ++k)
      for (int i = 0; i < pc.n; ++i) v[i] += __ldcs(ws + (int64_t)k * MN + base + i);
  }
}

__global__ void __launch_bounds__(kThreads)
    splitk_reduce_bf16_kernel(const float *__restrict__ ws, int splits, int64_t M, int64_t N,
                              uint16_t *__restrict__ C, int64_t ldc, uint32_t cpr, const ReduceTiles rt) {
  griddep_wait();  // the partials come from the GEMM launched just before
  const uint64_t t = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
  Piece pc;
  if (!reduce_piece(t, cpr, M, N, rt, &pc)) return;
  float v[4];
  sum_piece(ws, splits, rt.count ? (int64_t)rt.count * rt.rows * rt.cols : M * N,
            rt.count ? true : (N & 3) == 0, pc, v);
  uint16_t *dst = C + pc.r * ldc + pc.c;
  uint16_t h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat16 b = __float2bfloat16_rn(v[i]);  // round once, nearest even
    h[i] = *reinterpret_cast<const uint16_t *>(&b);
  }
  if (pc.n == 4 && (reinterpret_cast<uintptr_t>(dst) & 7) == 0) {
    *reinterpret_cast<uint2 *>(dst) = make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
  } else {
    for (int i = 0; i < pc.n; ++i) dst[i] = h[i];
  }
}

// int32 partials; stored as int32, or requantised to int16 / int8.
__global__ void __launch_bounds__(kThreads)
    splitk_reduce_s32_kernel(const int32_t *__restrict__ ws, int splits, int64_t M, int64_t N, void *__restrict__ C,
                             int64_t ldc, int out_bits, int shift, uint32_t cpr, const ReduceTiles rt) {
  griddep_wait();
  const uint64_t t = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
  Piece pc;
  if (!reduce_piece(t, cpr, M, N, rt, &pc)) return;
  int32_t v[4];
  sum_piece(ws, splits, rt.count ? (int64_t)rt.count * rt.rows * rt.cols : M * N,
            rt.count ? true : (N & 3) == 0, pc, v);
  if (out_bits == 32) {
    int32_t *dst = static_cast<int32_t *>(C) + pc.r * ldc + pc.c;
    if (pc.n == 4 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0)
      *reinterpret_cast<int4 *>(dst) = make_int4(v[0], v[1], v[2], v[3]);
    else
      for (int i = 0; i < pc.n; ++i) dst[i] = v[i];
    return;
  }
  const int32_t hi = (1 << (out_bits - 1)) - 1, lo = -hi - 1;
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = requantize_s32(v[i], shift, lo, hi);
  if (out_bits == 16) {
    int16_t *dst = static_cast<int16_t *>(C) + pc.r * ldc + pc.c;
    if (pc.n == 4 && (reinterpret_cast<uintptr_t>(dst) & 7) == 0)
      *reinterpret_cast<uint2 *>(dst) = make_uint2(((uint32_t)v[0] & 0xFFFFu) | ((uint32_t)v[1] << 16),
                                                   ((uint32_t)v[2] & 0xFFFFu) | ((uint32_t)v[3] << 16));
    else
      for (int i = 0; i < pc.n; ++i) dst[i] = (int16_t)v[i];
  } else {
    int8_t *dst = static_cast<int8_t *>(C) + pc.r * ldc + pc.c;
    if (pc.n == 4 && (reinterpret_cast<uintptr_t>(dst) & 3) == 0)
      *reinterpret_cast<uint32_t *>(dst) = ((uint32_t)v[0] & 0xFFu) | (((uint32_t)v[1] & 0xFFu) << 8) |
                                           (((uint32_t)v[2] & 0xFFu) << 16) | ((uint32_t)v[3] << 24);
    else
      for (int i = 0; i < pc.n; ++i) dst[i] = (int8_t)v[i];
  }
}

// One thread waits, with the GEMM kernels' bounded wait, on an mbarrier that
// nothing will ever arrive on: the wait gives up after limit_ns and records
// the timeout in the device error word, exactly as a stalled GEMM would.
__global__ void wait_timeout_probe_kernel(uint32_t *err, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_addr(&bar), 1);
    abort_flag = 0u;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) (void)mbar_wait(smem_addr(&bar), 0, &abort_flag, err, limit_ns);
}

// Reads n 16-byte vectors with streaming loads, four in flight per thread,
// and keeps nothing: the time of a plain read of that many bytes.  The
// result folds into one word that is written only if it equals a value no
// read of real data is expected to give, so the loads are not optimised away.
__global__ void __launch_bounds__(512) read_stream_kernel(const uint4 *__restrict__ p, uint64_t n, uint32_t *sink) {
  uint32_t acc = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n; i += 4 * stride) {
    const uint4 a = __ldcs(p + i), b = __ldcs(p + i + stride), c = __ldcs(p + i + 2 * stride),
                d = __ldcs(p + i + 3 * stride);
    acc ^= a.x ^ a.w ^ b.y ^ b.x ^ c.z ^ c.y ^ d.w ^ d.z;
  }
  for (; i < n; i += stride) {
    const uint4 a = __ldcs(p + i);
    acc ^= a.x ^ a.w;
  }
  if (acc == 0x9E3779B9u) *sink = acc;
}

}  // namespace

cudaError_t launch_read_stream(const void *p, size_t bytes, uint32_t *sink, int sms, cudaStream_t st) {
  const uint64_t n = bytes / 16;
  if (n == 0) return cudaSuccess;
  read_stream_kernel<<<(unsigned)(4 * sms), 512, 0, st>>>(static_cast<const uint4 *>(p), n, sink);
  return cudaGetLastError();
}

cudaError_t launch_wait_timeout_probe(uint32_t *err, uint64_t limit_ns, cudaStream_t st) {
  wait_timeout_probe_kernel<<<1, 32, 0, st>>>(err, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_s8_to_bf16_pair(const S8Job &a, const S8Job &b, int sms, cudaStream_t st) {
  (void)sms;  // both kernels cover their work with one thread per piece
  auto dense = [](const S8Job &j) {
    return j.ld_src == j.cols && j.ld_dst == j.cols && (reinterpret_cast<uintptr_t>(j.src) & 15) == 0 &&
           (reinterpret_cast<uintptr_t>(j.dst) & 15) == 0;
  };
  if (dense(a) && dense(b)) {
    const int64_t na = a.rows * a.cols, nb = b.rows * b.cols;
    const int64_t vecs = (na + 15) / 16 + (nb + 15) / 16;
    if (vecs == 0) return cudaSuccess;
    return launch_staging(s8_to_bf16_dense_kernel, vecs, st, a, b, na, nb);
  }
  const uint64_t cpr_a = (uint64_t)(a.cols + 15) / 16, cpr_b = (uint64_t)(b.cols + 15) / 16;
  const uint64_t items_a = (uint64_t)a.rows * cpr_a, items = items_a + (uint64_t)b.rows * cpr_b;
  if (items == 0) return cudaSuccess;
  return launch_staging(s8_to_bf16_pair_kernel, (int64_t)items, st, a, b, (uint32_t)(cpr_a ? cpr_a : 1),
                        (uint32_t)(cpr_b ? cpr_b : 1), items_a, items);
}

cudaError_t launch_pack_u16(const uint16_t *src, int64_t rows, int64_t cols, int64_t ld_src,
                            uint16_t *dst, int64_t ld_dst, int sms, cudaStream_t st) {
  (void)sms;
  const uint64_t cpr = (uint64_t)(cols + 7) / 8, items = (uint64_t)rows * cpr;
  if (items == 0) return cudaSuccess;
  return launch_staging(pack_u16_kernel, (int64_t)items, st, src, rows, cols, ld_src, dst, ld_dst, (uint32_t)cpr, items);
}

cudaError_t launch_zero_fill(void *C, int64_t M, int64_t N, int64_t ldc, int esize, int sms,
                             cudaStream_t st) {
  const int g = grid_for(M * N, 4, sms);
  if (esize == 1)
    zero_fill_kernel<uint8_t><<<g, kThreads, 0, st>>>(static_cast<uint8_t *>(C), M, N, ldc);
  else if (esize == 2)
    zero_fill_kernel<uint16_t><<<g, kThreads, 0, st>>>(static_cast<uint16_t *>(C), M, N, ldc);
  else
    zero_fill_kernel<int32_t><<<g, kThreads, 0, st>>>(static_cast<int32_t *>(C), M, N, ldc);
  return cudaGetLastError();
}

// Pieces (4 elements of a row) the reduction covers.
static uint64_t reduce_items(int64_t M, uint32_t cpr, const ReduceTiles &rt) {
  return rt.count == 0 ? (uint64_t)M * cpr : (uint64_t)rt.count * rt.rows * ((uint32_t)rt.cols / 4);
}

cudaError_t launch_splitk_reduce_bf16(const float *ws, int splits, int64_t M, int64_t N,
                                      uint16_t *C, int64_t ldc, const ReduceTiles &rt, cudaStream_t st) {
  const uint32_t cpr = (uint32_t)((N + 3) / 4);
  const uint64_t items = reduce_items(M, cpr, rt);
  return launch_ex(splitk_reduce_bf16_kernel, dim3((unsigned)((items + kThreads - 1) / kThreads)), dim3(kThreads),
                   0, st, 1, ws, splits, M, N, C, ldc, cpr, rt);
}

cudaError_t launch_splitk_reduce_s32(const int32_t *ws, int splits, int64_t M, int64_t N, void *C,
                                     int64_t ldc, int out_bits, int shift, const ReduceTiles &rt,
                                     cudaStream_t st) {
  const uint32_t cpr = (uint32_t)((N + 3) / 4);
  const uint64_t items = reduce_items(M, cpr, rt);
  return launch_ex(splitk_reduce_s32_kernel, dim3((unsigned)((items + kThreads - 1) / kThreads)), dim3(kThreads),
                   0, st, 1, ws, splits, M, N, C, ldc, out_bits, shift, cpr, rt);
}

}  // namespace gb300
