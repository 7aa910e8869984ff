// Algorithm 1 (the sketch) (Sec. 3): the sketch Y = Omega [A | b] in precision u_s.
//
//  * cast pass (Sec. 3.2 one-sided scaling): column maxima of [A | b] -> a
//    power-of-two exponent per column -> A_s = fl_s(2^k A) written K-major
//    (one row of Bt per column of A, contiguous over the m data rows), so
//    both tensor-core operands are K-major in 128-byte swizzled tiles.
//  * tcgen05 sketch: per CTA a 128-row slab of the sketch matrix, up to 512
//    columns of [A | b] in TMEM (FP32), a split of the m range.  Warp 0 feeds
//    Bt tiles by TMA, warp 1 issues tcgen05.mma (kind::f16 or kind::f8f6f4),
//    sixteen generator warps synthesise the sketch tile fl_s(G) in registers
//    and store it swizzled into shared memory, fixer warps settle the entries
//    that their estimate leaves open, and the generators drain TMEM into an FP32
//    partial per split.  G is never stored in global memory.
//  * CUDA-core sketch for u_s = F64 / F32 (no tensor-core format).
//  * reduce: FP64 sum of the split partials, times s^-1/2 and 2^-k_j.
#include <cudaTypedefs.h>

#include <cstring>
#include <type_traits>

#include "cast.cuh"
#include "common.cuh"
#include "gauss.cuh"
#include "kernels.h"

namespace lsq {

// ============================================================ omega test hook
template <int FMT>
__global__ void omega_kernel(int64_t s, int64_t j0, int64_t cols, uint32_t k0, uint32_t k1,
                             double* out) {
  const int64_t q_first = j0 >> 2, q_last = (j0 + cols - 1) >> 2;
  const int64_t nq = q_last - q_first + 1;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= s * nq) return;
  const int64_t i = idx / nq;
  const int64_t q = q_first + idx % nq;
  const uint4 x = philox4x32_10(gauss_counter((uint64_t)q, (uint32_t)i), k0, k1);
  double v[4];
  if constexpr (FMT == FMT_F64 || FMT == FMT_F32) {
    spec_gauss_pair(x.x, x.y, v[0], v[1]);
    spec_gauss_pair(x.z, x.w, v[2], v[3]);
    if constexpr (FMT == FMT_F32) {
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = (double)__double2float_rn(v[t]);
    }
  } else {
    uint32_t e0, o0, e1, o1;
    gauss_pair_bits<FMT>(x.x, x.y, e0, o0);
    gauss_pair_bits<FMT>(x.z, x.w, e1, o1);
    v[0] = bits_to_double<FMT>(e0);
    v[1] = bits_to_double<FMT>(o0);
    v[2] = bits_to_double<FMT>(e1);
    v[3] = bits_to_double<FMT>(o1);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int64_t j = q * 4 + t;
    if (j >= j0 && j < j0 + cols) out[i * cols + (j - j0)] = v[t];
  }
}

cudaError_t launch_omega(int fmt, int64_t s, int64_t j0, int64_t cols, uint64_t seed, double* out,
                         cudaStream_t st) {
  const int64_t nq = ((j0 + cols - 1) >> 2) - (j0 >> 2) + 1;
  const int64_t total = s * nq;
  const int threads = 256;
  const unsigned blocks = (unsigned)((total + threads - 1) / threads);
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  switch (fmt) {
    case FMT_F64: omega_kernel<FMT_F64><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    case FMT_F32: omega_kernel<FMT_F32><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    case FMT_F16: omega_kernel<FMT_F16><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    case FMT_BF16: omega_kernel<FMT_BF16><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    case FMT_E4M3: omega_kernel<FMT_E4M3><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    case FMT_BF16X3: omega_kernel<FMT_BF16><<<blocks, threads, 0, st>>>(s, j0, cols, k0, k1, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ============================================================ cast pass
// Roundings run on integer units (cast.cuh); the FP64 definition is left only
// for out-of-range values (subnormal results, overflow, subnormal or
// non-finite inputs).

// fl32(2^k x) as FP32 bits, x given by its FP64 bits: integer rounding, else the FP64
// definition (subnormal results, non-finite or subnormal x).
__device__ __forceinline__ uint32_t f32_scaled_bits(uint64_t u, int k) {
  uint32_t b;
  if (f64_scaled_to_f32_bits(u, k, b)) return b;   // normal x, 2^k x in FP32's range
  uint32_t t[3];
  if (cast_terms_int<EncF32>(u, k, t)) return t[0];
  return __float_as_uint(__double2float_rn(ldexp(__longlong_as_double((long long)u), k)));
}

// FP64 bits -> FP32 value, round to nearest even.
__device__ __forceinline__ float f64bits_to_f32(uint64_t u) {
  uint32_t b;
  if (f64_to_f32_bits(u, b)) return __uint_as_float(b);
  return __uint_as_float(f32_scaled_bits(u, 0));
}

__device__ __forceinline__ void colmax_a32_body(const double* __restrict__ A, int64_t lda,
                                                const double* __restrict__ b, int64_t m, int64_t n,
                                                unsigned long long* cmax, float* __restrict__ a32,
                                                int64_t lda32, int64_t rows_per_block, int* err, int64_t blk) {
  const int64_t r0 = blk * rows_per_block;
  const int64_t r1 = min(m, r0 + rows_per_block);
  const int64_t cend = a32 ? max(n + 1, lda32) : n + 1;
  const uint64_t* Au = reinterpret_cast<const uint64_t*>(A);
  const uint64_t* bu = reinterpret_cast<const uint64_t*>(b);
  constexpr uint64_t kAbs = 0x7FFFFFFFFFFFFFFFull;
  // |v| as FP64 bits is monotone in |v| for non-NaN values: the column maximum
  // is an integer maximum
  for (int64_t c = threadIdx.x; c < cend; c += blockDim.x) {
    uint64_t mx = 0;
    if (c < n) {
      int64_t i = r0;
      for (; i + 8 <= r1; i += 8) {   // eight loads in flight before any use
        uint64_t u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = __ldcs(Au + (i + q) * lda + c);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          mx = max(mx, u[q] & kAbs);
          if (a32) a32[(i + q) * lda32 + c] = f64bits_to_f32(u[q]);
        }
      }
      for (; i < r1; ++i) {
        const uint64_t u = __ldcs(Au + i * lda + c);
        mx = max(mx, u & kAbs);
        if (a32) a32[i * lda32 + c] = f64bits_to_f32(u);
      }
    } else if (c == n) {
      for (int64_t i = r0; i < r1; ++i) mx = max(mx, bu[i] & kAbs);
      if (a32 && c < lda32)
        for (int64_t i = r0; i < r1; ++i) a32[i * lda32 + c] = 0.0f;
    } else {
      for (int64_t i = r0; i < r1; ++i) a32[i * lda32 + c] = 0.0f;
    }
    if (c <= n && mx > 0) atomicMax(cmax + c, (unsigned long long)mx);
    // |v| bits at or above those of +infinity: an infinity or a NaN in the column
    if (c <= n && mx >= 0x7FF0000000000000ull) set_error(err, DEV_NONFINITE);
  }
}

__global__ void colmax_a32_kernel(const double* __restrict__ A, int64_t lda,
                                  const double* __restrict__ b, int64_t m, int64_t n,
                                  unsigned long long* cmax, float* __restrict__ a32, int64_t lda32,
                                  int64_t rows_per_block, int* err) {
  colmax_a32_body(A, lda, b, m, n, cmax, a32, lda32, rows_per_block, err, blockIdx.x);
}

cudaError_t launch_colmax_a32(const double* A, int64_t lda, const double* b, int64_t m, int64_t n,
                              unsigned long long* cmax_bits, float* a32, int64_t lda32, int* err,
                              cudaStream_t st) {
  const int64_t rows_per_block = 64;
  const unsigned blocks = (unsigned)((m + rows_per_block - 1) / rows_per_block);
  colmax_a32_kernel<<<blocks, 256, 0, st>>>(A, lda, b, m, n, cmax_bits, a32, lda32, rows_per_block, err);
  return cudaGetLastError();
}

__global__ void scale_exps_kernel(const unsigned long long* cmax, int64_t ncols, int t, int* kexp) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= ncols) return;
  const double mx = __longlong_as_double((long long)cmax[c]);
  int k = 0;
  if (t >= 0 && mx > 0.0 && isfinite(mx)) {
    int ex;
    frexp(mx, &ex);  // mx = f 2^ex, f in [0.5, 1)
    k = t - (ex - 1);
  }
  kexp[c] = k;
}

cudaError_t launch_scale_exps(const unsigned long long* cmax_bits, int64_t ncols, int t, int* kexp,
                              cudaStream_t st) {
  scale_exps_kernel<<<(unsigned)((ncols + 255) / 256), 256, 0, st>>>(cmax_bits, ncols, t, kexp);
  return cudaGetLastError();
}

template <int FMT>
struct FmtEnc;
template <>
struct FmtEnc<FMT_BF16> {
  using T = EncBF16;
};
template <>
struct FmtEnc<FMT_BF16X3> {
  using T = EncBF16;
};
template <>
struct FmtEnc<FMT_F16> {
  using T = EncF16;
};
template <>
struct FmtEnc<FMT_E4M3> {
  using T = EncE4M3;
};

// The terms of fl_s(2^k x) (x given by its FP64 bits u): integer path, else the
// FP64 definition (round-to-odd into FP32, then to the format).  BF16X3: the three
// BF16 terms of y = fl32(2^k x).
template <int FMT>
__device__ __forceinline__ void cast_bits(uint64_t u, int k, uint32_t (&t)[3]) {
  if constexpr (FMT == FMT_BF16X3) {
    split3_f32(f32_scaled_bits(u, k), t);
  } else if (!cast_terms_int<typename FmtEnc<FMT>::T>(u, k, t)) {
    t[0] = round_f64<FMT>(ldexp(__longlong_as_double((long long)u), k));
  }
}

// Bt layout: blocks of kBtBlock data rows; within a block, [plane][row][k] with
// rows = the padded columns of [A | b] (one row per column) and k contiguous, so a
// sketch CTA's K chunk of its column group lies in one contiguous stretch of a
// few MB (a K-major layout with m-long rows puts every row of a stage on its
// own page once m is in the millions).
//
// Single-term formats: tiles of 32 columns by as many rows as make 128 bytes of a column of
// Bt (64 rows; 128 for E4M3).  Each thread issues its loads of a column eight at a time and
// rounds on the high word (cast_hi; the general rounding of the few other values follows),
// the tile is transposed in its final format, and a warp stores 128 contiguous bytes.  Column
// tile fastest, as in the BF16X3 cast.  Bound by HBM (8 bytes read, 2 or 1 written a value):
// at 116 instructions an element and 32 x 32 tiles of 8-byte words it was bound by
// instruction issue (BF16, m = 1e5, n = 500: 201 us; now 87 us).
template <int FMT>
constexpr int kCastRows = FMT == FMT_E4M3 ? 128 : 64;
template <int FMT>
__device__ __forceinline__ void cast_transpose_body(const double* __restrict__ A, int64_t lda,
                                                    const double* __restrict__ b, int64_t m, int64_t n,
                                                    const int* __restrict__ kexp, void* __restrict__ Bt,
                                                    int64_t plane_rows, int64_t bx, int64_t by) {
  using F = typename FmtEnc<FMT>::T;
  using E = typename std::conditional<FMT == FMT_E4M3, uint8_t, uint16_t>::type;
  constexpr int ROWS = kCastRows<FMT>, VPW = 4 / (int)sizeof(E);
  __shared__ uint32_t tile[32][33];   // [column][row], VPW values a word, one word of padding
  const int64_t j0 = bx * ROWS, c0 = by * 32, c = c0 + threadIdx.x;
  const uint64_t* src = reinterpret_cast<const uint64_t*>(c < n ? A + c : b);
  const int64_t stride = c < n ? lda : 1;
  const int k = c <= n ? kexp[c] : 0;
  const CastRange cr = cast_range<F>(k);
  E* col = reinterpret_cast<E*>(tile[threadIdx.x]);
#pragma unroll
  for (int h = 0; h < ROWS / 64; ++h) {
    uint64_t u[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int64_t j = j0 + h * 64 + threadIdx.y + 8 * q;
      u[q] = (c <= n && j < m) ? __ldcs(src + j * stride) : 0ull;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t v;
      if (!cast_hi<F>(u[q], cr, v)) {
        uint32_t t[3];
        cast_bits<FMT>(u[q], k, t);
        v = t[0];
      }
      col[h * 64 + threadIdx.y + 8 * q] = (E)v;
    }
  }
  __syncthreads();
  const int64_t j = j0 + VPW * threadIdx.x, blk = j / kBtBlock, kk = j % kBtBlock;
  uint32_t* P = reinterpret_cast<uint32_t*>(Bt);
  for (int r = threadIdx.y; r < 32; r += 8)   // rows past column n and data rows past m: zeros
    if (c0 + r < plane_rows) P[((blk * plane_rows + c0 + r) * kBtBlock + kk) / VPW] = tile[r][threadIdx.x];
}

// BF16X3: y = fl32(2^k x) in three BF16 planes hi, lo, lo2 (same Bt layout).  Tiles of
// kCast3Rows rows x 32 columns.  y comes from the FP32 copy of A by a power-of-two
// scaling where that is exact (f32_scale_exact), else from the FP64 value (the b
// column, zeros, the bottom of FP32's range, or no FP32 copy); each thread writes two
// consecutive k of a row per plane, so a warp stores 128 contiguous bytes.
__device__ __forceinline__ void cast_bf16x3_body(const double* __restrict__ A, int64_t lda,
                                                 const double* __restrict__ b, const float* __restrict__ a32,
                                                 int64_t lda32, int64_t m, int64_t n,
                                                 const int* __restrict__ kexp, void* __restrict__ Bt,
                                                 int64_t plane_rows, int64_t bx, int64_t by) {
  __shared__ uint32_t tile[32][kCast3Rows + 1];   // [column][row]: y bits
  const int64_t j0 = bx * kCast3Rows, c0 = by * 32;
  const int64_t c = c0 + threadIdx.x;
  const int k = (c <= n) ? kexp[c] : 0;
  const uint64_t* Au = reinterpret_cast<const uint64_t*>(A);
  const uint64_t* bu = reinterpret_cast<const uint64_t*>(b);
  // the FP32 copy's values of the thread's column, all loads in flight before any use
  constexpr int kPer = kCast3Rows / 8;
  uint32_t av[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int64_t j = j0 + threadIdx.y + 8 * q;
    av[q] = (a32 != nullptr && c < n && j < m) ? __float_as_uint(__ldcs(a32 + j * lda32 + c)) : 0u;
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int r = threadIdx.y + 8 * q;
    const int64_t j = j0 + r;
    uint32_t y = 0;
    if (j < m && c <= n) {
      const bool done = a32 != nullptr && c < n && f32_scale_exact(av[q], k, y);
      if (!done) y = f32_scaled_bits(c < n ? __ldcs(Au + j * lda + c) : bu[j], k);
    }
    tile[threadIdx.x][r] = y;
  }
  __syncthreads();
  uint32_t* P = reinterpret_cast<uint32_t*>(Bt);   // pairs of BF16 values, k even first
  const int64_t pstride = plane_rows * kBtBlock / 2;
  const int64_t j = j0 + 2 * threadIdx.x;
  const int64_t blk = j / kBtBlock, kk = j % kBtBlock;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int64_t cc = c0 + r;
    if (cc >= plane_rows) continue;
    const int64_t base = ((blk * 3 * plane_rows + cc) * kBtBlock + kk) / 2;
    // the split of two values (cast.cuh: split3_f32) with the packed FP32 -> BF16 rounding
    float y0 = __uint_as_float(tile[r][2 * threadIdx.x]), y1 = __uint_as_float(tile[r][2 * threadIdx.x + 1]);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const uint32_t w = pack2<FMT_BF16>(y0, y1);
      P[base + t * pstride] = w;
      y0 = __fsub_rn(y0, __uint_as_float(w << 16));
      y1 = __fsub_rn(y1, __uint_as_float(w & 0xFFFF0000u));
    }
  }
}

// One-dimensional grid, column tile fastest: the column tiles of a row tile run together,
// so the 128-byte lines that neighbouring tiles share (rows of the FP32 copy need not start
// on a line) are read from DRAM once.
__global__ void cast_bf16x3_kernel(const double* __restrict__ A, int64_t lda, const double* __restrict__ b,
                                   const float* __restrict__ a32, int64_t lda32, int64_t m, int64_t n,
                                   const int* __restrict__ kexp, void* __restrict__ Bt, int64_t plane_rows) {
  const int64_t ct = (plane_rows + 31) / 32, id = blockIdx.x;
  cast_bf16x3_body(A, lda, b, a32, lda32, m, n, kexp, Bt, plane_rows, id / ct, id % ct);
}

template <int FMT>
__global__ void cast_transpose_kernel(const double* __restrict__ A, int64_t lda,
                                      const double* __restrict__ b, int64_t m, int64_t n,
                                      const int* __restrict__ kexp, void* __restrict__ Bt,
                                      int64_t plane_rows) {
  const int64_t ct = (plane_rows + 31) / 32, id = blockIdx.x;
  cast_transpose_body<FMT>(A, lda, b, m, n, kexp, Bt, plane_rows, id / ct, id % ct);
}

int64_t bt_blocks(int64_t m) { return (m + kBtBlock - 1) / kBtBlock; }

size_t bt_bytes(int fmt, int64_t m, int64_t plane_rows) {
  const int esz = (fmt == FMT_E4M3) ? 1 : 2;
  const int planes = (fmt == FMT_BF16X3) ? 3 : 1;
  return (size_t)bt_blocks(m) * planes * plane_rows * kBtBlock * esz;
}

int64_t cast_row_tiles(int fmt, int64_t m) {
  return bt_blocks(m) * kBtBlock / (fmt == FMT_BF16X3 ? kCast3Rows : fmt == FMT_E4M3 ? kCastRows<FMT_E4M3> : kCastRows<FMT_BF16>);
}

cudaError_t launch_cast_transpose(int fmt, const double* A, int64_t lda, const double* b, const float* a32,
                                  int64_t lda32, int64_t m, int64_t n, const int* kexp, void* Bt,
                                  int64_t plane_rows, cudaStream_t st) {
  if (plane_rows < n + 1) return cudaErrorInvalidValue;
  const int64_t tiles = cast_row_tiles(fmt, m) * ((plane_rows + 31) / 32);
  if (tiles > 2147483647LL) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)tiles;
  const dim3 block(32, 8);
  switch (fmt) {
    case FMT_F16: cast_transpose_kernel<FMT_F16><<<grid, block, 0, st>>>(A, lda, b, m, n, kexp, Bt, plane_rows); break;
    case FMT_BF16: cast_transpose_kernel<FMT_BF16><<<grid, block, 0, st>>>(A, lda, b, m, n, kexp, Bt, plane_rows); break;
    case FMT_E4M3: cast_transpose_kernel<FMT_E4M3><<<grid, block, 0, st>>>(A, lda, b, m, n, kexp, Bt, plane_rows); break;
    case FMT_BF16X3: cast_bf16x3_kernel<<<grid, block, 0, st>>>(A, lda, b, a32, lda32, m, n, kexp, Bt, plane_rows); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ============================================================ tcgen05 sketch
constexpr int kSkGenWarps = 16;
constexpr int kSkGenThreads = kSkGenWarps * 32;
// Fixers: two groups of warps take the stages in turn.  A double-float evaluation is a chain
// of about 1.4 us, so one group of two warps held every stage for that long (F16, m = 2e5,
// n = 1000, s = 3000: 1.73 ms, 1.75 us a stage).
constexpr int kSkFixGroups = 2;
constexpr int kSkFixWarps = 2;                // of a group
constexpr int kSkFixThreads = kSkFixWarps * 32;
constexpr int kSkFixFirst = 2 + kSkGenWarps;
constexpr int kSkQMax = 256;                 // undecided pairs queued per stage
constexpr size_t kSkSmem = 232448;           // the SM's shared memory: one CTA per SM
// Rings: three or four sketch tiles of 128 rows, and as many Bt slots as fit (at most
// kSkBRing).  A slot is one box of one plane (chunk rows), so a slot is refilled as soon as its
// own products are done, and the generators run up to four stages ahead.  Whole stages as
// slots (sketch tile and all boxes of Bt: 80 KB at 512 columns, so two of them) left both
// waiting for the refill's latency.  Rings, 128-byte rows and fixer groups together: BF16, m =
// 1e5, n = 500, s = 2000 459 -> 355 us (instruction issue of the generators), F16, m = 2e5, n =
// 1000, s = 3000 2.50 -> 1.65 ms, BF16X3, m = 2e5, n = 1000, s = 4000 4.99 -> 3.5 ms (tensor
// pipe 42 -> 59 %).
constexpr int sk_a_ring(int nt) { return nt == 1 ? 4 : 3; }
constexpr int kSkBRing = 16;
constexpr size_t kSkCtrl = 5120;             // barriers and queue counters (512 bytes), queues
static_assert(512 + sk_a_ring(1) * kSkQMax * 4 <= kSkCtrl, "a queue per sketch tile");
constexpr int kSkThreads = (2 + kSkGenWarps + kSkFixGroups * kSkFixWarps) * 32;   // TMA, MMA, generators, fixers

__device__ __forceinline__ void fix_barrier(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kSkFixThreads) : "memory");
}

// A stage is 128 bytes of K (64 elements of the 16-bit formats, 128 of E4M3): K-major
// operands in 128-byte rows, 128-byte swizzle.  (Stages of 64-byte rows for the three planes
// of BF16X3 issued twice the TMA rows and gave every generator thread a single Philox call.)
constexpr int kSkRowB = 128;

// Byte offset of 16-byte chunk kc of row `row` in a swizzled K-major tile.
__device__ __forceinline__ uint32_t swz_chunk(int row, int kc) {
  return (uint32_t)(row * kSkRowB + ((kc ^ (row & 7)) << 4));
}

// Y partial = fl_s(G)[128 rows] x (sum over NT planes of Bt)[bn columns] over one split of m.
//
// A stage passes through three groups of warps: the generators write the tile from FP32
// estimates and queue the pairs that the estimate leaves undecided (gauss.cuh); the fixers
// evaluate those in double-float and patch the tile while the generators are on the next stage;
// the MMA warp multiplies it.  So the GEMM always multiplies fl_s(G) itself.
//
// What bounds it: the generators' instruction issue where n is below about 500 a format
// term; beyond, a stage's way through generators, fixers and MMA with the refill of Bt (F16, n =
// 1000: issue 56 %, tensor pipe 30 % busy; BF16X3 37 % and 59 %).  (With the earlier FP32 estimate,
// 176 instructions a pair against 72 now, BF16, m = 1e5, n = 500, s = 2000 took 706 us.)  Before,
// the GEMM multiplied the estimates, kept lists of the undecided pairs and a second kernel
// evaluated them in FP64 and corrected the partials: 17 ms beside the GEMM's 17 ms for F16 at m = 1e6, n = 1000, s = 3000, a host round trip to see whether
// a list had overflowed, and in E4M3, whose subnormal range no estimate decided, always a
// second GEMM with every such pair in FP64 (131 ms at m = 6e5, n = 601, s = 1803).
//
// GROUPED: one launch for a batch of problems.  CTA b belongs to the problem p with
// grp.start[p] <= b < grp.start[p + 1]; its local index gives (tile, column group, split)
// in that problem's grid; the problem's arguments come from grp.tab[p] and its tensor map
// from grp.maps[p] (global memory, written by the host before the launch).
//
// SHARE (two column groups): the CTAs of the two column groups of a (tile, split) form a
// cluster and share the sketch operand: each generates and fixes half of the 128-row tile
// (rows 64 r .. 64 r + 63 for cluster rank r) in its own shared memory and copies it into its
// partner's stage with one bulk copy, completing the partner's full barrier; each MMA commit
// releases the stage in both CTAs (the empty barriers count two arrivals), so neither CTA
// overwrites a stage its partner still reads.  Before exiting, the producer waits for the
// last release of every stage, so no arrival from the partner can land in a CTA that has
// exited.
// Handing over (a.hand > 0): the (tile, split) items of a launch seldom fill whole waves of the
// SMs (two waves and a bit, by the rule for the splits), and shorter or longer splits would
// change the FP32 sums.  So the first a.hand items are each done by two CTAs: one takes the
// first steps, (k + 1) / (a.hand + 1) of them for item k, and leaves its accumulators in the item's
// place in `partial`; the other, among the last of the launch, loads them into TMEM and
// goes on.  The sums are those of one CTA, bit by bit.  The pieces' lengths are spread evenly
// over an item, so that all SMs finish together: first parts, whole items, second parts from
// the longest down.  Work is taken by ticket, so a second part waits (with a limit) only for a
// CTA that already runs and waits for nothing itself.  F16, m = 1e6, n = 1000, s = 3000 (2.2
// waves): 10.8 -> 8.2 ms.
template <int FMT, int NT, bool GROUPED, bool SHARE = false>
__global__ void __launch_bounds__(kSkThreads, 1)
    sketch_tc_kernel(const __grid_constant__ CUtensorMap tmB, const SketchTcArgs a_in, const SketchGroup grp) {
  static_assert(!SHARE || !GROUPED, "operand sharing runs for one problem");
  constexpr int GF = (FMT == FMT_BF16X3) ? FMT_BF16 : FMT;   // format of the sketch operand
  constexpr int EB = (GF == FMT_E4M3) ? 1 : 2;                // bytes per element
  constexpr int BK = kSkRowB / EB;                            // K elements per stage
  constexpr int EPC = 16 / EB;                                // elements per 16-byte chunk
  constexpr int CPR = kSkRowB / 16;                           // chunks per row
  constexpr int NCHUNK = 128 * CPR;                           // chunks per sketch tile
  constexpr int PPC = EPC / 2;                                // (a, b) pairs per chunk
  constexpr uint32_t S_BYTES = 128u * kSkRowB;
  constexpr int KSLICES = kSkRowB / 32;                         // MMA K slices (32 bytes) per stage
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t mt = blockIdx.x, ng = blockIdx.y, split = blockIdx.z;
  const CUtensorMap* tmp = &tmB;
  int gp = 0;
  if constexpr (GROUPED) {
    gp = group_of(grp.start, grp.nprob, blockIdx.x);
    const int64_t local = (int64_t)blockIdx.x - grp.start[gp];
    const int mtl = grp.tab[gp].mtiles, ngl = grp.tab[gp].ngroups;
    mt = local % mtl;
    ng = (local / mtl) % ngl;
    split = local / ((int64_t)mtl * ngl);
    tmp = grp.maps + gp;
  }
  const SketchTcArgs a = GROUPED ? grp.tab[gp] : a_in;
  constexpr int NA = sk_a_ring(NT), ROWB = kSkRowB;
  const int chunk = a.bn / a.nsub;
  const uint32_t slot_bytes = (uint32_t)chunk * ROWB;         // one box of one plane of Bt
  const int NB = min(kSkBRing, (int)((kSkSmem - 1024 - kSkCtrl - NA * S_BYTES) / slot_bytes));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 4 * NA + 2 * kSkBRing + 1);
  uint32_t* qcnt = tslot + 1;                                 // [NA]
  uint32_t* qbuf = reinterpret_cast<uint32_t*>(smem + 512);   // [NA][kSkQMax]
  uint8_t* ringA = smem + kSkCtrl;
  uint8_t* ringB = ringA + NA * S_BYTES;
  // sketch tiles -- afull: fixer warps (+ the partner's half); aempty: MMA commit (of both
  // CTAs, SHARE); genned: generator warps done with the estimates; fixed: undecided pairs
  // written and the queue reset.  Bt slots -- bfull: TMA bytes; bempty: MMA commit.
  const uint32_t afull0 = smem_u32(bars), aempty0 = smem_u32(bars + NA);
  const uint32_t genned0 = smem_u32(bars + 2 * NA), fixed0 = smem_u32(bars + 3 * NA);
  const uint32_t bfull0 = smem_u32(bars + 4 * NA), bempty0 = smem_u32(bars + 4 * NA + kSkBRing);
  const uint32_t done_bar = smem_u32(bars + 4 * NA + 2 * kSkBRing);

  constexpr uint32_t HALF = S_BYTES / 2;                      // the half tile a CTA generates (SHARE)
  constexpr int GCH = SHARE ? NCHUNK / 2 : NCHUNK;            // chunks this CTA generates per stage
  const uint32_t rank = SHARE ? cl_rank() : 0u;
  int piece = 0;                        // 1 and 2: first and second part of an item
  unsigned* piece_flag = nullptr;       // raised when the first part is in `partial`
  if constexpr (!GROUPED) {
    if (a.hand > 0) {
      volatile uint32_t* tick = reinterpret_cast<volatile uint32_t*>(smem + 508);   // behind qcnt
      if constexpr (SHARE) cl_sync();   // the partner runs
      if (threadIdx.x == 0 && rank == 0u) {
        const uint32_t t = atomicAdd(a.work, 1u);
        if constexpr (SHARE)
          asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cl_map(smem_u32(smem + 508), 1u)), "r"(t) : "memory");
        *tick = t;
      }
      if constexpr (SHARE) cl_sync();
      else __syncthreads();
      int64_t item = *tick;
      if (item < a.hand) {
        piece = 1;
      } else if (item >= a.items) {
        piece = 2;
        item -= a.items;
      }
      mt = item % a.mtiles;
      if constexpr (SHARE) {
        split = item / a.mtiles;
      } else {
        ng = (item / a.mtiles) % a.ngroups;
        split = item / ((int64_t)a.mtiles * a.ngroups);
      }
      if (piece) piece_flag = a.work + 1 + 2 * item + rank;
    }
  }
  int64_t k_begin = split * a.kchunk;
  const int64_t k_end = min(a.m, k_begin + a.kchunk);
  int nk = (int)((k_end - k_begin + BK - 1) / BK);
  if constexpr (!GROUPED) {
    if (piece) {
      const int64_t k = (int64_t)(piece_flag - (a.work + 1)) / 2;
      const int cut = min(nk, (int)((k + 1) * (a.kchunk / BK) / (a.hand + 1)));
      if (piece == 1) {
        nk = cut;
      } else {
        k_begin += (int64_t)cut * BK;
        nk -= cut;
        if (cut == 0) piece = 0;   // no first part
      }
      if (nk == 0) return;   // nothing to do, or to go on with (every thread of the cluster)
    }
  }

  if (threadIdx.x == 0) {
    for (int st = 0; st < NA; ++st) {
      mbar_init(afull0 + 8 * st, kSkFixWarps);
      mbar_init(aempty0 + 8 * st, SHARE ? 2 : 1);
      mbar_init(genned0 + 8 * st, kSkGenWarps);
      mbar_init(fixed0 + 8 * st, kSkFixWarps);
      qcnt[st] = 0;
    }
    for (int sl = 0; sl < NB; ++sl) {
      mbar_init(bfull0 + 8 * sl, 1);
      mbar_init(bempty0 + 8 * sl, 1);
    }
    mbar_init(done_bar, 1);
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tslot), (uint32_t)a.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tslot;
  if (!GROUPED && piece == 2) {   // the first part's accumulators, as the epilogue left them
    if (warp >= 2 && warp < kSkFixFirst) {
      if (lane == 0) {
        auto raised = [&]() {
          unsigned f;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(piece_flag) : "memory");
          return f != 0u;
        };
        if (!raised()) {
          const uint64_t t0 = globaltimer_ns();
          while (!raised()) {
            if (globaltimer_ns() - t0 > kWaitLimitNs) {
              set_error(a.err, DEV_TIMEOUT_GRID);
              break;
            }
          }
        }
      }
      __syncwarp();
      const int q = warp & 3;
      const int64_t i = mt * 128 + q * 32 + lane;
      for (int c0 = 32 * ((warp - 2) >> 2); c0 < a.bn; c0 += 32 * (kSkGenWarps / 4)) {
        uint32_t r[32];
#pragma unroll
        for (int cc = 0; cc < 32; ++cc) {
          const int64_t col = ng * a.bn + c0 + cc;
          r[cc] = (i < a.s && c0 + cc < a.bn && col < a.ncols)
                      ? __float_as_uint(__ldcg(a.partial + (split * a.ncols + col) * a.s_pad + i))
                      : 0u;
        }
        tmem_st_32x32b_x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
      }
      tmem_st_wait();
      tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
  }
  if constexpr (SHARE) cl_sync();   // the partner's barriers are initialised before any copy or commit

  // Pair pi of chunk kc, row `row` of a sketch tile: its words drawn again, fl_s(G) stored.
  auto resolve_pair = [&](uint8_t* S, int row, int kc, int pi, int64_t kbase) {
    const uint64_t q = ((uint64_t)(kbase + kc * EPC) >> 2) + (uint64_t)(pi >> 1);
    const uint4 x = philox4x32_10(gauss_counter(q, (uint32_t)(mt * 128 + row)), a.k0, a.k1);
    uint32_t be, bo;
    gauss_pair_resolve<GF>((pi & 1) ? x.z : x.x, (pi & 1) ? x.w : x.y, be, bo);
    uint8_t* cp = S + swz_chunk(row, kc);
    if constexpr (EB == 2)
      *reinterpret_cast<uint32_t*>(cp + 4 * pi) = be | (bo << 16);
    else
      *reinterpret_cast<uint16_t*>(cp + 2 * pi) = (uint16_t)(be | (bo << 8));
  };

  if (warp == 0) {
    // ---------------- TMA producer: NT planes x nsub boxes of [chunk rows x 128 bytes]
    if (lane == 0) {
      if constexpr (GROUPED) {   // the map was written through the generic proxy
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                         reinterpret_cast<uint64_t>(tmp))
                     : "memory");
      }
      prefetch_tmap(tmp);
      int sl = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int ks = 0; ks < nk && ok; ++ks) {
        const int64_t kx = k_begin + (int64_t)ks * BK;
        const int32_t kin = (int32_t)(kx % kBtBlock), kblk = (int32_t)(kx / kBtBlock);
        for (int c = 0; c < a.nsub && ok; ++c)
          for (int t = 0; t < NT; ++t) {
            ok = mbar_wait(bempty0 + 8 * sl, ph ^ 1u, a.err, DEV_TIMEOUT_EMPTY);
            if (!ok) break;
            mbar_arrive_expect_tx(bfull0 + 8 * sl, slot_bytes);
            tma_load_3d(smem_u32(ringB) + (uint32_t)sl * slot_bytes, tmp, kin,
                        (int32_t)(t * a.rows_per_plane + ng * a.bn + c * chunk), kblk, bfull0 + 8 * sl);
            if (++sl == NB) {
              sl = 0;
              ph ^= 1u;
            }
          }
      }
      if constexpr (SHARE) {
        // tail: the last release of every sketch tile (both MMAs) has arrived here
        for (int st = 0; st < NA && st < nk; ++st) {
          const int last = st + ((nk - 1 - st) / NA) * NA;
          if (!mbar_wait(aempty0 + 8 * st, (uint32_t)(last / NA) & 1u, a.err, DEV_TIMEOUT_EMPTY)) break;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      const uint32_t idesc = make_idesc(GF == FMT_BF16 ? 1u : 0u, 128u, (uint32_t)chunk);
      int sl = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int ks = 0; ks < nk && ok; ++ks) {
        const int st = ks % NA;
        ok = mbar_wait(afull0 + 8 * st, (uint32_t)(ks / NA) & 1u, a.err, DEV_TIMEOUT_FULL);
        if (!ok) break;
        const uint32_t sa = smem_u32(ringA) + (uint32_t)st * S_BYTES;
        for (int c = 0; c < a.nsub && ok; ++c) {
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            ok = mbar_wait(bfull0 + 8 * sl, ph, a.err, DEV_TIMEOUT_FULL);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sb = smem_u32(ringB) + (uint32_t)sl * slot_bytes;
#pragma unroll
            for (int kk = 0; kk < KSLICES; ++kk) {
              const uint64_t ad = sw128_desc(sa + kk * 32), bd = sw128_desc(sb + kk * 32);
              const uint32_t acc = (ks | kk | t | (piece & 2)) != 0 ? 1u : 0u;
              if constexpr (GF == FMT_E4M3)
                mma_f8(tmem_base + (uint32_t)(c * chunk), ad, bd, idesc, acc);
              else
                mma_f16(tmem_base + (uint32_t)(c * chunk), ad, bd, idesc, acc);
            }
            tc_commit(bempty0 + 8 * sl);
            if (++sl == NB) {
              sl = 0;
              ph ^= 1u;
            }
          }
        }
        if constexpr (SHARE) tc_commit_mc(aempty0 + 8 * st, (uint16_t)0x3);
        else tc_commit(aempty0 + 8 * st);
      }
      tc_commit(done_bar);
    }
  } else if (warp < kSkFixFirst) {
    // ---------------- generator warps: fl_s(G) tile, 128 rows x BK columns
    const int g = threadIdx.x - 64;
    for (int ks = 0; ks < nk; ++ks) {
      const int st = ks % NA;
      const uint32_t ph = (uint32_t)(ks / NA) & 1u;
      if (!mbar_wait(aempty0 + 8 * st, ph ^ 1u, a.err, DEV_TIMEOUT_EMPTY)) break;
      if (!mbar_wait(fixed0 + 8 * st, ph ^ 1u, a.err, DEV_TIMEOUT_EMPTY)) break;
      uint8_t* S = ringA + st * S_BYTES;
      const int64_t kbase = k_begin + (int64_t)ks * BK;
      // One 16-byte chunk (HPI Philox calls, PPC pairs) per item.  No branch until every pair of
      // the thread is estimated: the calls interleave, and und collects the undecided pairs.
      constexpr int HPI = EPC / 4;
      constexpr int IPT = (GCH + kSkGenThreads - 1) / kSkGenThreads;   // items per thread
      static_assert(GCH % kSkGenThreads == 0 && IPT * PPC <= 32, "whole items, one bit per pair");
      uint32_t und = 0;
#pragma unroll
      for (int it = 0; it < IPT; ++it) {
        const int c = g + it * kSkGenThreads;
        const int row = c / CPR + (int)rank * 64, kc = c % CPR;
        const uint32_t i = (uint32_t)(mt * 128 + row);
        const uint64_t q0 = (uint64_t)(kbase + kc * EPC) >> 2;
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < HPI; ++h) {
          const uint4 x = philox4x32_10(gauss_counter(q0 + h, i), a.k0, a.k1);
          uint32_t p0, p1;   // the two pairs of the call, packed
          const bool ok0 = gauss_pair_est<GF>(x.x, x.y, p0);
          const bool ok1 = gauss_pair_est<GF>(x.z, x.w, p1);
          und |= (ok0 ? 0u : 1u << (it * PPC + 2 * h)) | (ok1 ? 0u : 2u << (it * PPC + 2 * h));
          if constexpr (EB == 2) {
            w[2 * h] = p0;
            w[2 * h + 1] = p1;
          } else {
            w[h] = p0 | (p1 << 16);
          }
        }
        *reinterpret_cast<uint4*>(S + swz_chunk(row, kc)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      while (und != 0u) {
        const int bit = __ffs((int)und) - 1;
        und &= und - 1u;
        const int c = g + (bit / PPC) * kSkGenThreads;
        const int row = c / CPR + (int)rank * 64, kc = c % CPR, pi = bit % PPC;
        const uint32_t slot = atomicAdd(qcnt + st, 1u);
        if (slot < (uint32_t)kSkQMax)
          qbuf[st * kSkQMax + slot] = ((uint32_t)row << 8) | ((uint32_t)kc << 4) | (uint32_t)pi;
        else   // queue full: resolve in place
          resolve_pair(S, row, kc, pi, kbase);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(genned0 + 8 * st);
    }
  } else {
    // ---------------- fixer warps: the queued pairs of a stage, overlapping the generation
    // of the next one
    const int group = (warp - kSkFixFirst) / kSkFixWarps;
    const int fx = threadIdx.x - (kSkFixFirst + group * kSkFixWarps) * 32;
    for (int ks = group; ks < nk; ks += kSkFixGroups) {
      const int st = ks % NA;
      const uint32_t ph = (uint32_t)(ks / NA) & 1u;
      if (!mbar_wait(genned0 + 8 * st, ph, a.err, DEV_TIMEOUT_FULL)) break;
      uint8_t* S = ringA + st * S_BYTES;
      const int64_t kbase = k_begin + (int64_t)ks * BK;
      const uint32_t nq = min(qcnt[st], (uint32_t)kSkQMax);
      for (uint32_t qi = fx; qi < nq; qi += kSkFixThreads) {
        const uint32_t pos = qbuf[st * kSkQMax + qi];
        resolve_pair(S, (int)(pos >> 8), (int)((pos >> 4) & 15), (int)(pos & 15), kbase);
      }
      fence_proxy_async_smem();
      fix_barrier(group);       // the group has read qcnt and written its pairs
      if (fx == 0) {
        qcnt[st] = 0;
        if constexpr (SHARE) {   // the finished half tile: whole rows, one contiguous run
          const uint32_t src = smem_u32(S) + rank * HALF;
          bulk_s2s(cl_map(src, rank ^ 1u), src, HALF, cl_map(afull0 + 8 * st, rank ^ 1u));
        }
      }
      __syncwarp();
      if (lane == 0) {
        if (SHARE && fx == 0) mbar_arrive_expect_tx(afull0 + 8 * st, HALF);   // the partner's half
        else mbar_arrive(afull0 + 8 * st);
        mbar_arrive(fixed0 + 8 * st);
      }
    }
  }

  // ---------------- epilogue: the generator warps drain TMEM, four warps to each quarter of
  // its lanes (a warp reaches lanes 32 (warp % 4) ..), 32 columns at a time
  if (warp >= 2 && warp < kSkFixFirst) {
    mbar_wait(done_bar, 0, a.err, DEV_TIMEOUT_DONE);
    tc_fence_after();
    const int q = warp & 3;
    const int64_t i = mt * 128 + q * 32 + lane;
    for (int c0 = 32 * ((warp - 2) >> 2); c0 < a.bn; c0 += 32 * (kSkGenWarps / 4)) {
      uint32_t r[32];
      tmem_ld_32x32b_x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, r);
      tmem_ld_wait();
      if (i < a.s) {
#pragma unroll
        for (int cc = 0; cc < 32; ++cc) {
          const int64_t col = ng * a.bn + c0 + cc;
          if (c0 + cc < a.bn && col < a.ncols)
            a.partial[(split * a.ncols + col) * a.s_pad + i] = __uint_as_float(r[cc]);
        }
      }
    }
  }
  tc_fence_before();
  if (!GROUPED && piece == 1) __threadfence();
  __syncthreads();
  if (!GROUPED && piece == 1 && threadIdx.x == 0) atomicExch(piece_flag, 1u);
  if constexpr (SHARE) cl_sync();   // neither CTA leaves while its partner may still copy or commit into it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)a.tmem_cols);
  }
}

static int round_up_int(int64_t v, int64_t q) { return (int)(((v + q - 1) / q) * q); }

bool plan_sketch_tc(int fmt, int64_t s, int64_t m, int64_t ncols, int num_sms, SketchPlan* p,
                    int64_t max_kchunk) {
  if (fmt != FMT_F16 && fmt != FMT_BF16 && fmt != FMT_E4M3 && fmt != FMT_BF16X3) return false;
  const int EB = (fmt == FMT_E4M3) ? 1 : 2;
  p->nt = (fmt == FMT_BF16X3) ? 3 : 1;
  p->rowb = (p->nt == 3) ? 64 : 128;
  const int BK = kSkRowB / EB;   // the kernel's K step
  p->fmt = fmt;
  p->s = s;
  p->m = m;
  p->ncols = ncols;
  p->ngroups = (int)((ncols + 511) / 512);
  int bn = round_up_int((ncols + p->ngroups - 1) / p->ngroups, 16);
  if (bn > 256) {
    bn = round_up_int(bn, 32);
    p->nsub = 2;
  } else {
    p->nsub = 1;
  }
  p->bn = bn;
  p->mtiles = (int)((s + 127) / 128);
  const size_t stage = (size_t)128 * p->rowb + (size_t)p->nt * bn * p->rowb;
  // the ring the plan guarantees room for: whole stages of rowb-byte rows, at least two (the
  // kernel lays out its rings in the SM's whole shared memory)
  p->stages = (4 * stage + 1024 + 512 + 4 * kSkQMax * 12 <= 232448) ? 4 : 2;
  p->smem = 1024 + (size_t)p->stages * stage + 512 + (size_t)p->stages * kSkQMax * 12;
  if (p->smem > 232448) return false;
  const int64_t base = (int64_t)p->mtiles * p->ngroups;
  const int64_t ksteps = (m + BK - 1) / BK;
  int64_t splits = (2 * (int64_t)num_sms + base - 1) / base;
  if (splits < 1) splits = 1;
  if (splits > ksteps) splits = ksteps;
  int64_t steps_per = (ksteps + splits - 1) / splits;
  if (max_kchunk == 0 && fmt == FMT_BF16X3) {
    // Single precision on BF16 tensor cores: the FP32 accumulation of one split,
    // not the cast, limits Y once the split is long (the error of the sum grows
    // about linearly with its length, so kappa(A R^-1) does too: 378 at 8e5 rows,
    // 6.8 at 8192 and 3.5 at 2048 for m = 4e6, n = 1000, kappa(A) = 1e7).  Splits of
    // at most kBf16x3Chunk rows, unless their FP32 partials would pass kPartialBudget.
    constexpr int64_t kBf16x3Chunk = 2048;
    constexpr double kPartialBudget = 34359738368.0;   // 32 GiB
    const double per_split = 4.0 * (double)ncols * (double)s;
    const int64_t max_splits = (int64_t)(kPartialBudget / per_split);
    int64_t want = (m + kBf16x3Chunk - 1) / kBf16x3Chunk;
    // at most 25 % more splits, so that the grid fills its last wave of CTAs best
    int64_t best = want, best_idle = -1;
    for (int64_t w = want; w <= want + want / 4; ++w) {
      const int64_t ctas = base * w, waves = (ctas + num_sms - 1) / num_sms;
      const int64_t idle = waves * num_sms - ctas;
      if (best_idle < 0 || idle < best_idle) {
        best = w;
        best_idle = idle;
      }
    }
    want = best;
    if (want > max_splits) want = max_splits;
    if (want > 65535) want = 65535;
    if (want > splits) {
      const int64_t sp = (ksteps + want - 1) / want;
      if (sp < steps_per) steps_per = sp;
    }
  }
  if (max_kchunk > 0) {
    const int64_t cap_steps = max_kchunk / BK > 0 ? max_kchunk / BK : 1;
    if (steps_per > cap_steps) steps_per = cap_steps;
  }
  p->kchunk = steps_per * BK;
  p->splits = (int)((m + p->kchunk - 1) / p->kchunk);
  p->s_pad = s;
  return true;
}

bool encode_bt_tmap(CUtensorMap* tm, const void* Bt, int fmt, int64_t rows, int64_t m, int box_rows) {
  // looked up once (thread-safe static initialisation; batched solves call this
  // from several host threads)
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }();
  if (!fn) return false;
  const int EB = (fmt == FMT_E4M3) ? 1 : 2;
  static_assert(kBtBlock % kSkRowB == 0, "a stage never straddles two blocks");
  // (k within the block, row over all planes, block)
  cuuint64_t dims[3] = {(cuuint64_t)kBtBlock, (cuuint64_t)rows, (cuuint64_t)bt_blocks(m)};
  cuuint64_t strides[2] = {(cuuint64_t)(kBtBlock * EB), (cuuint64_t)(rows * kBtBlock * EB)};
  cuuint32_t box[3] = {(cuuint32_t)(kSkRowB / EB), (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(tm, EB == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                  const_cast<void*>(Bt), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// The number of items to hand over, for `slots` CTAs (or pairs) at a time: none where the items fill
// their waves to within kSkHandSteps K steps an SM (two more starts of the pipeline and the
// accumulators' way through L2 take about 20 us, a step 0.35 us or more).
constexpr int kSkHandSteps = 64;
int sketch_hand_items(int64_t items, int64_t steps, int64_t slots) {
  if (slots < 2 || items < slots || items % slots == 0) return 0;
  const int64_t idle = slots - items % slots;
  return steps * idle / slots >= kSkHandSteps && slots - 1 <= kSkHandMax ? (int)(slots - 1) : 0;
}

template <int FMT, int NT>
static cudaError_t launch_tc_inst(const SketchPlan& p, const CUtensorMap& tm, SketchTcArgs a,
                                  unsigned* work, cudaStream_t st) {
  dim3 grid((unsigned)p.mtiles, (unsigned)p.ngroups, (unsigned)p.splits);
  const SketchGroup none{};
  const int64_t steps = p.kchunk / (kSkRowB / (p.fmt == FMT_E4M3 ? 1 : 2));
  auto plan_hand = [&](int64_t items, int slots) -> cudaError_t {
    a.hand = sketch_hand_items(items, steps, slots);
    if (a.hand == 0) return cudaSuccess;
    a.items = (int)items;
    a.work = work;
    grid.x = (unsigned)(items + a.hand);
    grid.z = 1;
    return cudaMemsetAsync(work, 0, (1 + 2 * (size_t)a.hand) * sizeof(unsigned), st);
  };
  if (p.ngroups == 2) {
    // the two column groups of a (tile, split) share the generated operand (a cluster of two)
    auto kern = sketch_tc_kernel<FMT, NT, false, true>;
    cudaError_t e = allow_dyn_smem(kern, kSkSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kSkThreads);
    cfg.dynamicSmemBytes = kSkSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 2;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int pairs = 0;
    if (steps >= kSkHandSteps) {
      e = cudaOccupancyMaxActiveClusters(&pairs, kern, &cfg);
      if (e == cudaSuccess) e = plan_hand((int64_t)p.mtiles * p.splits, pairs);
      if (e != cudaSuccess) return e;
      cfg.gridDim = grid;
    }
    return cudaLaunchKernelEx(&cfg, kern, tm, a, none);
  }
  auto kern = sketch_tc_kernel<FMT, NT, false>;
  cudaError_t e = allow_dyn_smem(kern, kSkSmem);
  if (e != cudaSuccess) return e;
  if (steps >= kSkHandSteps) {
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = plan_hand((int64_t)p.mtiles * p.ngroups * p.splits, sms);
    if (e != cudaSuccess) return e;
    if (a.hand) grid.y = 1;
  }
  kern<<<grid, kSkThreads, kSkSmem, st>>>(tm, a, none);
  return cudaGetLastError();
}

template <int FMT, int NT>
static cudaError_t launch_tc_grouped_inst(const SketchGroup& g, int64_t ctas, cudaStream_t st) {
  auto kern = sketch_tc_kernel<FMT, NT, true>;
  cudaError_t e = allow_dyn_smem(kern, kSkSmem);
  if (e != cudaSuccess) return e;
  CUtensorMap unused;
  std::memset(&unused, 0, sizeof(unused));
  kern<<<(unsigned)ctas, kSkThreads, kSkSmem, st>>>(unused, SketchTcArgs{}, g);
  return cudaGetLastError();
}

cudaError_t launch_sketch_tc(const SketchPlan& p, const CUtensorMap& tm, uint64_t seed,
                             float* partial, unsigned* work, int* err, cudaStream_t st) {
  const SketchTcArgs a = sketch_tc_args(p, seed, partial, err);
  switch (p.fmt) {
    case FMT_F16: return launch_tc_inst<FMT_F16, 1>(p, tm, a, work, st);
    case FMT_BF16: return launch_tc_inst<FMT_BF16, 1>(p, tm, a, work, st);
    case FMT_E4M3: return launch_tc_inst<FMT_E4M3, 1>(p, tm, a, work, st);
    case FMT_BF16X3: return launch_tc_inst<FMT_BF16X3, 3>(p, tm, a, work, st);
  }
  return cudaErrorInvalidValue;
}

SketchTcArgs sketch_tc_args(const SketchPlan& p, uint64_t seed, float* partial, int* err) {
  SketchTcArgs a{};
  a.s = p.s;
  a.m = p.m;
  a.ncols = p.ncols;
  a.kchunk = p.kchunk;
  a.s_pad = p.s_pad;
  a.bn = p.bn;
  a.nsub = p.nsub;
  a.rows_per_plane = p.ngroups * p.bn;
  a.mtiles = p.mtiles;
  a.ngroups = p.ngroups;
  int tc = 32;
  while (tc < p.bn) tc <<= 1;
  a.tmem_cols = tc;
  a.k0 = (uint32_t)seed;
  a.k1 = (uint32_t)(seed >> 32);
  a.partial = partial;
  a.err = err;
  return a;
}

cudaError_t launch_sketch_tc_grouped(int fmt, const SketchGroup& g, int64_t ctas, cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  if (ctas > 2147483647LL) return cudaErrorInvalidValue;
  switch (fmt) {
    case FMT_F16: return launch_tc_grouped_inst<FMT_F16, 1>(g, ctas, st);
    case FMT_BF16: return launch_tc_grouped_inst<FMT_BF16, 1>(g, ctas, st);
    case FMT_E4M3: return launch_tc_grouped_inst<FMT_E4M3, 1>(g, ctas, st);
    case FMT_BF16X3: return launch_tc_grouped_inst<FMT_BF16X3, 3>(g, ctas, st);
  }
  return cudaErrorInvalidValue;
}

// The pairs of one split a generator warp can leave undecided (4 * kchunk pairs a warp, with a
// margin over the fractions in gauss.cuh), and the number of generator warps of the grid.
uint32_t sketch_rec_cap(const SketchPlan& p) {
  const int64_t pairs = 4 * p.kchunk;
  const int64_t div = (p.fmt == FMT_F16) ? 16 : (p.fmt == FMT_E4M3) ? 1024 : 128;
  return (uint32_t)(pairs / div + 64);
}
int64_t sketch_rec_lists(const SketchPlan& p) {
  return (int64_t)p.mtiles * p.ngroups * p.splits * kSkGenWarps;
}

// ============================================================ CUDA-core sketch
// CTA tile: 16 sketch rows x 256 columns of [A | b]; K step 16; 256 threads,
// each 4 rows x 4 columns.  The sketch tile is generated once per K step.
template <typename T>
__global__ void __launch_bounds__(256)
    sketch_cc_kernel(const double* __restrict__ A, int64_t lda, const double* __restrict__ b,
                     int64_t m, int64_t n, int64_t s, uint32_t k0, uint32_t k1, int64_t kchunk,
                     T* __restrict__ partial, int64_t s_pad) {
  constexpr int BM = 16, BN = 256, BKc = 16;
  __shared__ T Gs[BKc][BM];
  __shared__ T Bs[BKc][BN];
  const int tid = threadIdx.x;
  const int64_t i0 = (int64_t)blockIdx.x * BM, c0 = (int64_t)blockIdx.y * BN;
  const int64_t split = blockIdx.z;
  const int64_t kb = split * kchunk, ke = min(m, kb + kchunk);
  const int tr = (tid >> 6) * 4, tc = (tid & 63) * 4;
  T acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = T(0);
  for (int64_t k = kb; k < ke; k += BKc) {
    // sketch tile: 16 rows x 16 K -> 64 Philox calls (4 K each)
    if (tid < 64) {
      const int r = tid >> 2, qq = tid & 3;
      const int64_t j = k + qq * 4;
      const uint4 x = philox4x32_10(gauss_counter((uint64_t)j >> 2, (uint32_t)(i0 + r)), k0, k1);
      double v[4];
      spec_gauss_pair(x.x, x.y, v[0], v[1]);
      spec_gauss_pair(x.z, x.w, v[2], v[3]);
#pragma unroll
      for (int t = 0; t < 4; ++t) Gs[qq * 4 + t][r] = (T)v[t];  // T = float rounds to nearest
    }
    for (int e = tid; e < BKc * BN; e += 256) {
      const int kk = e / BN, cc = e % BN;
      const int64_t j = k + kk, c = c0 + cc;
      double v = 0.0;
      if (j < ke) {
        if (c < n) v = A[j * lda + c];
        else if (c == n) v = b[j];
      }
      Bs[kk][cc] = (T)v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BKc; ++kk) {
      T gv[4], bv[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) gv[x] = Gs[kk][tr + x];
#pragma unroll
      for (int y = 0; y < 4; ++y) bv[y] = Bs[kk][tc + y];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fma(gv[x], bv[y], acc[x][y]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const int64_t c = c0 + tc + y;
    if (c > n) continue;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int64_t i = i0 + tr + x;
      if (i < s) partial[(split * (n + 1) + c) * s_pad + i] = acc[x][y];
    }
  }
}

cudaError_t launch_sketch_cc(int fmt, const double* A, int64_t lda, const double* b, int64_t m,
                             int64_t n, int64_t s, uint64_t seed, int splits, int64_t kchunk,
                             void* partial, int64_t s_pad, cudaStream_t st) {
  dim3 grid((unsigned)((s + 15) / 16), (unsigned)((n + 1 + 255) / 256), (unsigned)splits);
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  if (fmt == FMT_F64)
    sketch_cc_kernel<double><<<grid, 256, 0, st>>>(A, lda, b, m, n, s, k0, k1, kchunk,
                                                   static_cast<double*>(partial), s_pad);
  else if (fmt == FMT_F32)
    sketch_cc_kernel<float><<<grid, 256, 0, st>>>(A, lda, b, m, n, s, k0, k1, kchunk,
                                                  static_cast<float*>(partial), s_pad);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

// ============================================================ split reduce
// FP64 partials: an FP64 sum.  FP32 partials (the tensor-core splits): Knuth's TwoSum
// in FP32, an error-free transformation of each addition, with the rounding errors
// collected in a second FP32 word; hi + lo carries the sum of the splits to about
// 2^-48 relative (double-float), on the FP32 pipe instead of GB300's narrow FP64 pipe
// (the sum over thousands of 2048-row splits at m = 4e6 is 8e9 additions).
template <typename TP>
__device__ __forceinline__ void sketch_reduce_body(const TP* __restrict__ partial, int splits, int64_t ncols,
                                                   int64_t s, int64_t s_pad, const int* __restrict__ kexp,
                                                   double inv_sqrt_s, double* __restrict__ Y, int64_t bx,
                                                   int64_t c) {
  const int64_t i = bx * (int64_t)blockDim.x + threadIdx.x;
  if (i >= s) return;
  double acc;
  if constexpr (sizeof(TP) == 8) {
    acc = 0.0;
    for (int sp = 0; sp < splits; ++sp) acc += (double)partial[((int64_t)sp * ncols + c) * s_pad + i];
  } else {
    float hi = 0.0f, lo = 0.0f;
    const TP* p = partial + c * s_pad + i;
    const int64_t stride = ncols * s_pad;
    for (int sp = 0; sp < splits; ++sp) {
      const float x = __ldcs(p + (int64_t)sp * stride);
      const float t = __fadd_rn(hi, x);
      const float xb = __fsub_rn(t, hi);
      const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, xb)), __fsub_rn(x, xb));
      hi = t;
      lo = __fadd_rn(lo, err);
    }
    acc = (double)hi + (double)lo;
  }
  const int k = kexp ? kexp[c] : 0;
  Y[c * s + i] = ldexp(acc * inv_sqrt_s, -k);
}

template <typename TP>
__global__ void sketch_reduce_kernel(const TP* __restrict__ partial, int splits, int64_t ncols,
                                     int64_t s, int64_t s_pad, const int* __restrict__ kexp,
                                     double inv_sqrt_s, double* __restrict__ Y) {
  sketch_reduce_body<TP>(partial, splits, ncols, s, s_pad, kexp, inv_sqrt_s, Y, blockIdx.x, blockIdx.y);
}

// ============================================================ grouped (batched) forms
// One launch per stage for a batch of problems: CTA b works for the problem p with
// start[p] <= b < start[p + 1] (start: prefix sums of the per-problem CTA counts), on
// the block of that problem's own grid given by b - start[p].  Per-problem arguments
// come from a device table.
__global__ void grouped_colmax_kernel(const GCast* __restrict__ tab, const int* __restrict__ start, int nprob,
                                      int* err) {
  const int p = group_of(start, nprob, blockIdx.x);
  const GCast& g = tab[p];
  colmax_a32_body(g.A, g.lda, g.b, g.m, g.n, g.cmax, g.a32, g.lda32, kGroupedColmaxRows, err,
                  (int64_t)blockIdx.x - start[p]);
}

__global__ void grouped_scale_exps_kernel(const GCast* __restrict__ tab, const int* __restrict__ start,
                                          int nprob, int t) {
  const int p = group_of(start, nprob, blockIdx.x);
  const GCast& g = tab[p];
  const int64_t c = ((int64_t)blockIdx.x - start[p]) * blockDim.x + threadIdx.x;
  if (c > g.n) return;
  const double mx = __longlong_as_double((long long)g.cmax[c]);
  int k = 0;
  if (t >= 0 && mx > 0.0 && isfinite(mx)) {
    int ex;
    frexp(mx, &ex);
    k = t - (ex - 1);
  }
  g.kexp[c] = k;
}

template <int FMT>
__global__ void grouped_cast_kernel(const GCast* __restrict__ tab, const int* __restrict__ start, int nprob) {
  const int p = group_of(start, nprob, blockIdx.x);
  const GCast& g = tab[p];
  const int64_t local = (int64_t)blockIdx.x - start[p], ct = (g.plane_rows + 31) / 32;   // column tile fastest
  if constexpr (FMT == FMT_BF16X3)
    cast_bf16x3_body(g.A, g.lda, g.b, g.a32, g.lda32, g.m, g.n, g.kexp, g.Bt, g.plane_rows, local / ct, local % ct);
  else
    cast_transpose_body<FMT>(g.A, g.lda, g.b, g.m, g.n, g.kexp, g.Bt, g.plane_rows, local / ct, local % ct);
}

__global__ void grouped_sketch_reduce_kernel(const GReduce* __restrict__ tab, const int* __restrict__ start,
                                             int nprob) {
  const int p = group_of(start, nprob, blockIdx.x);
  const GReduce& g = tab[p];
  const int64_t local = (int64_t)blockIdx.x - start[p];
  const int64_t gx = (g.s + 255) / 256;
  sketch_reduce_body<float>(g.partial, g.splits, g.ncols, g.s, g.s_pad, g.kexp, 1.0 / sqrt((double)g.s), g.Y,
                            local % gx, local / gx);
}

cudaError_t launch_grouped_cast(int fmt, const GCast* tab, const int* colmax_start, int64_t colmax_ctas,
                                const int* exps_start, int64_t exps_ctas, const int* cast_start,
                                int64_t cast_ctas, int nprob, int t, int* err, cudaStream_t st) {
  if (colmax_ctas > 2147483647LL || cast_ctas > 2147483647LL) return cudaErrorInvalidValue;
  grouped_colmax_kernel<<<(unsigned)colmax_ctas, 256, 0, st>>>(tab, colmax_start, nprob, err);
  grouped_scale_exps_kernel<<<(unsigned)exps_ctas, 256, 0, st>>>(tab, exps_start, nprob, t);
  const int planes = (fmt == FMT_BF16X3) ? 3 : 1;
  const dim3 block(32, 8);
  switch (fmt) {
    case FMT_F16: grouped_cast_kernel<FMT_F16><<<(unsigned)cast_ctas, block, 0, st>>>(tab, cast_start, nprob); break;
    case FMT_BF16: grouped_cast_kernel<FMT_BF16><<<(unsigned)cast_ctas, block, 0, st>>>(tab, cast_start, nprob); break;
    case FMT_E4M3: grouped_cast_kernel<FMT_E4M3><<<(unsigned)cast_ctas, block, 0, st>>>(tab, cast_start, nprob); break;
    case FMT_BF16X3: grouped_cast_kernel<FMT_BF16X3><<<(unsigned)cast_ctas, block, 0, st>>>(tab, cast_start, nprob); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_grouped_sketch_reduce(const GReduce* tab, const int* start, int64_t ctas, int nprob,
                                         cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  grouped_sketch_reduce_kernel<<<(unsigned)ctas, 256, 0, st>>>(tab, start, nprob);
  return cudaGetLastError();
}

cudaError_t launch_sketch_reduce(const void* partial, bool partial_f64, int splits, int64_t ncols,
                                 int64_t s, int64_t s_pad, const int* kexp, double* Y,
                                 cudaStream_t st) {
  dim3 grid((unsigned)((s + 255) / 256), (unsigned)ncols);
  const double inv = 1.0 / sqrt((double)s);
  if (partial_f64)
    sketch_reduce_kernel<double><<<grid, 256, 0, st>>>(static_cast<const double*>(partial), splits,
                                                       ncols, s, s_pad, kexp, inv, Y);
  else
    sketch_reduce_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float*>(partial), splits,
                                                      ncols, s, s_pad, kexp, inv, Y);
  return cudaGetLastError();
}

}  // namespace lsq
