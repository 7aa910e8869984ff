// Streaming passes over A and the small kernels of LSQR and FGMRES (Alg. 2).
//
// Passes (one coalesced, 128-bit vectorised read of A per call, a warp per
// row, the row kept in registers for both products):
//   LSQR (Alg. 2, LSQR start):  q = A t + cu u ; P = A^T q ; sum q^2
//   FGMRES (Alg. 2, FGMRES):  w_top = v_top + A z_bot ; P = A^T v_top
//   residual (refinement, u_r):  f = b - r - A x ; P = A^T (-r)
// P is reduced per CTA (fixed order) and then across CTAs by colsum, so the
// results are deterministic.
#include <type_traits>

#include <algorithm>

#include "common.cuh"
#include "batch.h"
#include "iter.h"
#include "kernels.h"
#include "trsv.cuh"

namespace lsq {

// ============================================================ block helpers
__device__ __forceinline__ double block_sum_d(double v, double* red) {
  v = warp_sum(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
  if (warp == 0) t = warp_sum(t);
  if (threadIdx.x == 0) red[32] = t;
  __syncthreads();
  return red[32];
}


template <typename T, int VW>
struct VecOf;
template <>
struct VecOf<float, 4> {
  using type = float4;
};
template <>
struct VecOf<double, 2> {
  using type = double2;
};
template <>
struct VecOf<double, 1> {
  using type = double;
};

template <typename T, int VW>
__device__ __forceinline__ void load_vec(const T* p, T (&o)[VW], bool streaming) {
  using V = typename VecOf<T, VW>::type;
  V v = streaming ? __ldcs(reinterpret_cast<const V*>(p)) : *reinterpret_cast<const V*>(p);
  const T* e = reinterpret_cast<const T*>(&v);
#pragma unroll
  for (int k = 0; k < VW; ++k) o[k] = e[k];
}

// The register form, for rows the bulk ring does not take (odd or unaligned FP64 strides, FP64
// beyond 800 columns).  Every lane works on all VPL vectors, padding included: tests that leave out
// the vectors past the row (as the other forms have for FP64) cost it 2 to 10 % at every width
// (residual, m = 60,000 with an odd stride: n = 187 112 us without, 124 with; n = 256 116, 125).
template <typename T, int VW, int VPL, int MODE>
__device__ __forceinline__ void pass_body(PassArgs<T> p, int64_t blk, int64_t nblk) {
  if (p.done && *p.done) return;
  if (p.jp) {
    const int64_t j = *p.jp;
    p.x += j * p.xstr;
    p.v += j * p.vstr;
  }
  extern __shared__ __align__(16) unsigned char pass_smem[];
  T* red = reinterpret_cast<T*>(pass_smem);          // [8 warps][nv * VW]
  __shared__ double sqred[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = blk * 8 + warp, tw = nblk * 8;
  T xv[VPL][VW], acc[VPL][VW];
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int idx = lane + 32 * v;
    if (idx < p.nv) {
      load_vec<T, VW>(p.x + (int64_t)idx * VW, xv[v], false);
    } else {
      for (int k = 0; k < VW; ++k) xv[v][k] = T(0);
    }
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[v][k] = T(0);
  }
  T cu = T(0);
  if (MODE == PM_LSQR) cu = (T)((p.cu_ptr ? *p.cu_ptr : 1.0) * p.cu_mul);
  double sqacc = 0.0;   // lane 0: q^2 in FP64
  for (int64_t i = gw; i < p.m; i += 2 * tw) {
    const int64_t i2 = i + tw;
    const bool has2 = i2 < p.m;
    T a[VPL][VW], a2[VPL][VW];
    const T* row = p.A + i * p.lda;
    const T* row2 = p.A + i2 * p.lda;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int idx = lane + 32 * v;
      if (idx < p.nv) {
        load_vec<T, VW>(row + (int64_t)idx * VW, a[v], true);
      } else {
        for (int k = 0; k < VW; ++k) a[v][k] = T(0);
      }
      if (has2 && idx < p.nv) {
        load_vec<T, VW>(row2 + (int64_t)idx * VW, a2[v], true);
      } else {
        for (int k = 0; k < VW; ++k) a2[v][k] = T(0);
      }
    }
    T d = 0, d2 = 0;
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int k = 0; k < VW; ++k) {
        d = fma(a[v][k], xv[v][k], d);
        d2 = fma(a2[v][k], xv[v][k], d2);
      }
    warp_sum2(d, d2);
    T c1, c2 = T(0);
    if (MODE == PM_LSQR) {
      const T q = d + cu * p.uin[i];
      c1 = q;
      if (lane == 0) {
        p.uout[i] = q;
        sqacc = fma((double)q, (double)q, sqacc);
      }
      if (has2) {
        const T q2 = d2 + cu * p.uin[i2];
        c2 = q2;
        if (lane == 0) {
          p.uout[i2] = q2;
          sqacc = fma((double)q2, (double)q2, sqacc);
        }
      }
    } else if (MODE == PM_FGM) {
      c1 = p.v[i];
      if (lane == 0) p.az[i] = d;
      if (has2) {
        c2 = p.v[i2];
        if (lane == 0) p.az[i2] = d2;
      }
    } else {
      const double ri = p.r[i];
      c1 = (T)(-ri);
      if (lane == 0) p.f[i] = (p.b[i] - ri) - (double)d;
      if (has2) {
        const double ri2 = p.r[i2];
        c2 = (T)(-ri2);
        if (lane == 0) p.f[i2] = (p.b[i2] - ri2) - (double)d2;
      }
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
      for (int k = 0; k < VW; ++k) acc[v][k] = fma(c1, a[v][k], fma(c2, a2[v][k], acc[v][k]));
  }
  // CTA reduction of acc (fixed order over warps)
  const int width = p.nv * VW;
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int idx = lane + 32 * v;
    if (idx < p.nv) {
      for (int k = 0; k < VW; ++k) red[warp * width + idx * VW + k] = acc[v][k];
    }
  }
  if (MODE == PM_LSQR && lane == 0) sqred[warp] = sqacc;
  __syncthreads();
  for (int c = threadIdx.x; c < p.n; c += blockDim.x) {
    T s = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w * width + c];
    p.Pblk[blk * p.n + c] = s;
  }
  if (MODE == PM_LSQR && threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += sqred[w];
    p.sq[blk] = s;
  }
}

// The pass of the grouped launches (rows of at most 64 float4 or 256 doubles): the body
// above with each warp's rows streamed through a ring of its own in shared memory, kRingPairs
// row pairs ahead with asynchronous copies.  A lane copies and reads the same pieces, so the
// ring needs no barrier.  Two rows a warp in flight, as the register form has, left HBM waiting
// (381 us an FGMRES pass and 480 us an LSQR pass over 1.8 GB); now 288 and 384 (with 3 or 4 pairs
// fewer CTAs fit an SM: 2 % and 1 % more for a batch of 32).  FP64 residual, 3.6 GB: 3.98 ms, 2.9 now
// (1.4 of them FMAs).
constexpr int kRingPairs = 2;
template <typename T, int VW, int VPL, int MODE>
__device__ __forceinline__ void pass_ring_body(PassArgs<T> p, int64_t blk, int64_t nblk) {
  constexpr int CB = VW * (int)sizeof(T);   // bytes of a copy
  static_assert(CB == 16 || CB == 8, "asynchronous copies");
  if (p.done && *p.done) return;
  if (p.jp) {
    const int64_t j = *p.jp;
    p.x += j * p.xstr;
    p.v += j * p.vstr;
  }
  extern __shared__ __align__(16) unsigned char pass_smem[];
  __shared__ double sqred[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = blk * 8 + warp, tw = nblk * 8;
  const int width = p.nv * VW;
  T* ring = reinterpret_cast<T*>(pass_smem) + (size_t)warp * 2 * kRingPairs * width;
  const int nvl = (p.nv + 31) >> 5;   // vectors a lane uses
  T xv[VPL][VW], acc[VPL][VW];
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int idx = lane + 32 * v;
    if (idx < p.nv) {
      load_vec<T, VW>(p.x + (int64_t)idx * VW, xv[v], false);
    } else {
      for (int k = 0; k < VW; ++k) xv[v][k] = T(0);
    }
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[v][k] = T(0);
  }
  const T cu = (MODE == PM_LSQR) ? (T)((p.cu_ptr ? *p.cu_ptr : 1.0) * p.cu_mul) : T(0);
  // rows i and i + tw into slots 2 s and 2 s + 1
  auto fetch = [&](int64_t i, int s) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int64_t row = i + e * tw;
      if (row < p.m) {
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int idx = lane + 32 * v;
          if (idx < p.nv) {
            const uint32_t dst = smem_u32(ring + (size_t)(2 * s + e) * width + idx * VW);
            const T* src = p.A + row * p.lda + (int64_t)idx * VW;
            if constexpr (CB == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
          }
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < kRingPairs; ++s) fetch(gw + 2 * s * tw, s);
  // q^2 is summed in FP64, 32 rows at a time: lane l keeps the q of the rows l, l + 32, ... of the
  // warp's sequence (an FP64 product per row is one more serial step of 67 cycles)
  double sqacc = 0.0;
  T qkeep = T(0);
  int qn = 0, slot = 0;
  for (int64_t i = gw; i < p.m; i += 2 * tw) {
    const int64_t i2 = i + tw;
    const bool has2 = i2 < p.m;
    T s0, s1 = T(0), b0 = T(0), b1 = T(0);
    if constexpr (MODE == PM_RES) {
      s0 = (T)p.r[i];
      b0 = (T)p.b[i];
      if (has2) {
        s1 = (T)p.r[i2];
        b1 = (T)p.b[i2];
      }
    } else {
      const T* sv = MODE == PM_LSQR ? p.uin : p.v;
      s0 = sv[i];
      if (has2) s1 = sv[i2];
    }
    asm volatile("cp.async.wait_group %0;" ::"n"(kRingPairs - 1) : "memory");
    const T* ra = ring + (size_t)(2 * slot) * width;
    const T* rb = ra + width;
    // a row's pieces: zero past its end (and for a second row that is none)
    auto pieces = [&](int v, T (&a)[VW], T (&a2)[VW]) {
      const int idx = lane + 32 * v;
#pragma unroll
      for (int k = 0; k < VW; ++k) a[k] = a2[k] = T(0);
      if (idx < p.nv) {
        load_vec<T, VW>(ra + idx * VW, a, false);
        if (has2) load_vec<T, VW>(rb + idx * VW, a2, false);
      }
    };
    T d = T(0), d2 = T(0);
#pragma unroll
    for (int v = 0; v < VPL; ++v)
      if (sizeof(T) == 4 || v < nvl) {
        T a[VW], a2[VW];
        pieces(v, a, a2);
#pragma unroll
        for (int k = 0; k < VW; ++k) {
          d = fma(a[k], xv[v][k], d);
          d2 = fma(a2[k], xv[v][k], d2);
        }
      }
    warp_sum2(d, d2);
    T c1, c2;
    if constexpr (MODE == PM_LSQR) {
      c1 = d + cu * s0;
      c2 = has2 ? d2 + cu * s1 : T(0);
      if (lane == 0) p.uout[i] = c1;
      if (lane == qn) qkeep = c1;
      if (has2) {
        if (lane == 0) p.uout[i2] = c2;
        if (lane == qn + 1) qkeep = c2;
      }
      qn += 2;
      if (qn == 32) {
        sqacc = fma((double)qkeep, (double)qkeep, sqacc);
        qkeep = T(0);
        qn = 0;
      }
    } else if constexpr (MODE == PM_FGM) {
      c1 = s0;
      c2 = s1;
      if (lane == 0) p.az[i] = d;
      if (lane == 0 && has2) p.az[i2] = d2;
    } else {
      c1 = -s0;
      c2 = -s1;
      if (lane == 0) p.f[i] = (b0 - s0) - d;
      if (lane == 0 && has2) p.f[i2] = (b1 - s1) - d2;
    }
    // the pieces again from the ring: held in registers over the sum they would cost a CTA an SM
    asm volatile("" ::: "memory");
#pragma unroll
    for (int v = 0; v < VPL; ++v)
      if (sizeof(T) == 4 || v < nvl) {
        T a[VW], a2[VW];
        pieces(v, a, a2);
#pragma unroll
        for (int k = 0; k < VW; ++k) acc[v][k] = fma(c1, a[k], fma(c2, a2[k], acc[v][k]));
      }
    fetch(i + 2 * kRingPairs * tw, slot);
    slot = slot + 1 == kRingPairs ? 0 : slot + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  // CTA reduction of acc (fixed order over warps), each warp's sums in its own ring
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int idx = lane + 32 * v;
    if (idx < p.nv)
      for (int k = 0; k < VW; ++k) ring[idx * VW + k] = acc[v][k];
  }
  if (MODE == PM_LSQR) {
    sqacc = warp_sum(fma((double)qkeep, (double)qkeep, sqacc));
    if (lane == 0) sqred[warp] = sqacc;
  }
  __syncthreads();
  const T* all = reinterpret_cast<const T*>(pass_smem);
  for (int c = threadIdx.x; c < p.n; c += blockDim.x) {
    T s = T(0);
#pragma unroll
    for (int w = 0; w < 8; ++w) s += all[(size_t)w * 2 * kRingPairs * width + c];
    p.Pblk[blk * p.n + c] = s;
  }
  if (MODE == PM_LSQR && threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += sqred[w];
    p.sq[blk] = s;
  }
}

template <typename T, int VW, int VPL, int MODE>
__global__ void __launch_bounds__(256) pass_kernel(PassArgs<T> p) {
  pass_body<T, VW, VPL, MODE>(p, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------ bulk-streamed passes
// A producer warp streams stages of 16 consecutive rows of A into a shared-memory
// ring with cp.async.bulk (completion on an mbarrier).  FP32 (bound by HBM): sixteen consumer
// warps take a row of each stage.  FP64 (bound by its pipe; the
// rates: common.cuh): eight warps take two rows, whose sums share a reduction (five additions instead of ten), in one chain of FMAs; with a row a
// warp and four interleaved chains, n = 187 took 38 us at m = 20011 (FGMRES) and n = 500
// 274 us at m = 1e5 (residual); now 27 and 240.  Each CTA owns a contiguous range of rows.
// The per-row scalars of the next stage are loaded one stage ahead.
//   PM_LSQR: q = A t + cu u ; u_out = q ; P = A^T q ; sq = sum q^2
//   PM_FGM : az = A z ; P = A^T v            (v_top + az is formed by the Arnoldi step)
//   PM_RES : f = b - r - A x ; P = A^T (-r)
constexpr int kBulkRows = 16;
template <typename T>
constexpr int kBulkRw = sizeof(T) == 8 ? 2 : 1;                          // rows of a warp
template <typename T>
constexpr int kBulkThreads = (kBulkRows / kBulkRw<T> + 1) * 32;

template <typename T>
struct BulkArgs {
  const T* A;
  int64_t lda, m;
  int n, nv, stages;
  int64_t rows_per_cta;
  const T* x;                  // multiplied vector (nv * VW entries, zero padded)
  const int* jp;               // FGM: x and v are column (*jp) of their bases
  int64_t xstr, vstr;
  const T* uin;                // LSQR
  T* uout;
  const double* cu_ptr;
  double cu_mul;
  const double* sq_ref;        // SCALED: a norm that the size of q goes with
  const T* v;                  // FGM coefficient vector
  T* az;
  const double* r;             // RES
  const double* b;
  double* f;
  T* Pblk;
  double* sq;
  const int* done;
  int* err;
};

// 2^-e for ref in [2^e, 2^(e + 1)), |e| <= 126; 1 for 0 and non-finite ref
__device__ __forceinline__ float pow2_near_inverse(double ref) {
  const int e = (int)((__double_as_longlong(ref) >> 52) & 0x7FF);
  return e == 0 || e == 0x7FF ? 1.0f : __uint_as_float((uint32_t)(127 - min(126, max(-126, e - 1023))) << 23);
}

template <typename T, int VW, int VPL, int MODE, bool SCALED = false>
__global__ void __launch_bounds__(kBulkThreads<T>, 1) pass_bulk_kernel(BulkArgs<T> p) {
  if (p.done && *p.done) return;
  if (MODE == PM_FGM && p.jp) {
    const int64_t j = *p.jp;
    p.x += j * p.xstr;
    p.v += j * p.vstr;
  }
  extern __shared__ __align__(128) unsigned char bulk_smem[];
  const uint32_t stage_bytes = (uint32_t)(kBulkRows * p.lda * sizeof(T));
  uint64_t* bars = reinterpret_cast<uint64_t*>(bulk_smem + (size_t)p.stages * stage_bytes);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + p.stages);
  constexpr int RW = kBulkRw<T>, CW = kBulkRows / RW;   // rows of a warp, consumer warps
  __shared__ double sqred[CW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = (int64_t)blockIdx.x * p.rows_per_cta;
  const int64_t r1 = min(p.m, r0 + p.rows_per_cta);
  const int nst = r0 < r1 ? (int)((r1 - r0 + kBulkRows - 1) / kBulkRows) : 0;
  if (threadIdx.x == 0) {
    for (int k = 0; k < p.stages; ++k) {
      mbar_init(full0 + 8 * k, 1);
      mbar_init(empty0 + 8 * k, CW);
    }
    fence_barrier_init();
  }
  __syncthreads();
  T acc[VPL][VW];
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int k = 0; k < VW; ++k) acc[v][k] = T(0);
  // Sum of q^2.  FP64: 32 rows at a time, as in pass_ring_body.  FP32: in single (FP64 sums cost this form
  // 10 to 40 %: n = 600, m = 1e6 400 us, 565); SCALED, for the start's residual, which has the scale
  // of b: of q times a power of two, since squares of |q| above 1.8e19 or below 1e-23 leave the range.
  // (An instantiation of its own: the product cost the iterations' passes up to 4 %.)
  constexpr bool WIDE = sizeof(T) == 8;
  T sqacc = T(0), qkeep = T(0);
  const float qs = SCALED ? pow2_near_inverse(*p.sq_ref) : 1.0f;
  if (warp == CW) {
    // ---------------- producer
    if (lane == 0) {
      const uint64_t pol = l2_policy_evict_first();   // A is read once per pass
      for (int it = 0; it < nst; ++it) {
        const int slot = it % p.stages;
        const uint32_t ph = (uint32_t)(it / p.stages) & 1u;
        if (!mbar_wait(empty0 + 8 * slot, ph ^ 1u, p.err, DEV_TIMEOUT_EMPTY)) break;
        const int64_t row0 = r0 + (int64_t)it * kBulkRows;
        const int rows = (int)min((int64_t)kBulkRows, r1 - row0);
        const uint32_t bytes = (uint32_t)(rows * p.lda * sizeof(T));
        mbar_arrive_expect_tx(full0 + 8 * slot, bytes);
        bulk_load_hint(smem_u32(bulk_smem + (size_t)slot * stage_bytes), p.A + row0 * p.lda, bytes,
                       full0 + 8 * slot, pol);
      }
    }
  } else {
    // ---------------- consumers: warp `warp` takes rows RW warp .. RW warp + RW - 1 of every stage
    const int nvl = (p.nv + 31) >> 5;   // vectors a lane uses
    T xv[VPL][VW];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int idx = lane + 32 * v;
      if (idx < p.nv) {
        load_vec<T, VW>(p.x + (int64_t)idx * VW, xv[v], false);
      } else {
        for (int k = 0; k < VW; ++k) xv[v][k] = T(0);
      }
    }
    const T cu = (MODE == PM_LSQR) ? (T)((p.cu_ptr ? *p.cu_ptr : 1.0) * p.cu_mul) : T(0);
    // per-row scalars for a window of 32 stages: lane l holds the scalars of stage
    // base + l; the next window is loaded while the current one is consumed
    // scalars in the pass precision (no FP64 conversions in the FP32 passes)
    using S = typename std::conditional<MODE == PM_RES, double, T>::type;
    auto load_window = [&](int base, S (&s0)[RW], S (&s1)[RW]) {
      const int it = base + lane;
#pragma unroll
      for (int e = 0; e < RW; ++e) {
        const int64_t row = r0 + (int64_t)it * kBulkRows + warp * RW + e;
        s0[e] = S(0);
        s1[e] = S(0);
        if (it < nst && row < r1) {
          if constexpr (MODE == PM_LSQR) s0[e] = p.uin[row];
          if constexpr (MODE == PM_FGM) s0[e] = p.v[row];
          if constexpr (MODE == PM_RES) {
            s0[e] = p.r[row];
            s1[e] = p.b[row];
          }
        }
      }
    };
    S w0[RW], w1[RW], x0n[RW], x1n[RW];
    load_window(0, w0, w1);
    load_window(32, x0n, x1n);
    for (int it = 0; it < nst; ++it) {
      if ((it & 31) == 0 && it > 0) {
#pragma unroll
        for (int e = 0; e < RW; ++e) {
          w0[e] = x0n[e];
          w1[e] = x1n[e];
        }
        load_window(it + 32, x0n, x1n);
      }
      S c0[RW], c1s[RW];
#pragma unroll
      for (int e = 0; e < RW; ++e) {
        c0[e] = __shfl_sync(0xffffffffu, w0[e], it & 31);
        c1s[e] = (MODE == PM_RES) ? __shfl_sync(0xffffffffu, w1[e], it & 31) : S(0);
      }
      const int slot = it % p.stages;
      const uint32_t ph = (uint32_t)(it / p.stages) & 1u;
      if (!mbar_wait(full0 + 8 * slot, ph, p.err, DEV_TIMEOUT_FULL)) break;
      const int64_t row = r0 + (int64_t)it * kBulkRows + warp * RW;
      if (row < r1) {
        const bool has2 = RW == 2 && row + 1 < r1;   // a missing second row counts as zeros
        const T* srow = reinterpret_cast<const T*>(bulk_smem + (size_t)slot * stage_bytes) + warp * RW * p.lda;
        T a[RW == 1 ? VPL : 1][VW];   // FP32 keeps the row; FP64 (pipe-bound) reads it again for A^T
        // vector v of row e of the warp
        auto row_vec = [&](int e, int v, T (&o)[VW]) {
          const int idx = lane + 32 * v;
          if (idx < p.nv && (e == 0 || has2)) {
            load_vec<T, VW>(srow + e * p.lda + idx * VW, o, false);
          } else {
            for (int k = 0; k < VW; ++k) o[k] = T(0);
          }
        };
        T d[RW];
        if constexpr (RW == 1) {
#pragma unroll
          for (int v = 0; v < VPL; ++v) row_vec(0, v, a[v]);
          // four interleaved chains: in LSQR the row's A^T q update waits on this sum
          T dq[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
          for (int v = 0; v < VPL; ++v)
#pragma unroll
            for (int k = 0; k < VW; ++k)
              dq[(v * VW + k) & 3] = fma(a[v][k], xv[v][k], dq[(v * VW + k) & 3]);
          d[0] = warp_sum((dq[0] + dq[1]) + (dq[2] + dq[3]));
        } else {
          d[0] = T(0);
          d[RW - 1] = T(0);
#pragma unroll
          for (int v = 0; v < VPL; ++v)
            if (v < nvl) {
              T y0[VW], y1[VW];
              row_vec(0, v, y0);
              row_vec(1, v, y1);
#pragma unroll
              for (int k = 0; k < VW; ++k) {
                d[0] = fma(y0[k], xv[v][k], d[0]);
                d[RW - 1] = fma(y1[k], xv[v][k], d[RW - 1]);
              }
            }
          warp_sum2(d[0], d[RW - 1]);
        }
        T coef[RW];
#pragma unroll
        for (int e = 0; e < RW; ++e) {
          const bool in = e == 0 || has2;
          if (MODE == PM_LSQR) {
            const T q = d[e] + cu * (T)c0[e];
            coef[e] = q;
            if (lane == 0 && in) {
              p.uout[row + e] = q;
              if constexpr (!WIDE) {
                const float qe = SCALED ? q * qs : q;
                sqacc = fmaf(qe, qe, sqacc);
              }
            }
            if (WIDE && lane == ((it * RW) & 31) + e && in) qkeep = q;
          } else if (MODE == PM_FGM) {
            coef[e] = (T)c0[e];
            if (lane == 0 && in) p.az[row + e] = d[e];
          } else {
            coef[e] = (T)(-c0[e]);
            if (lane == 0 && in) p.f[row + e] = (c1s[e] - c0[e]) - (double)d[e];
          }
        }
        if (MODE == PM_LSQR && WIDE && ((it + 1) * RW & 31) == 0) {
          sqacc = fma(qkeep, qkeep, sqacc);
          qkeep = T(0);
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v)
          if constexpr (RW == 1) {
#pragma unroll
            for (int k = 0; k < VW; ++k) acc[v][k] = fma(coef[0], a[v][k], acc[v][k]);
          } else if (v < nvl) {
            T y0[VW], y1[VW];
            row_vec(0, v, y0);
            row_vec(1, v, y1);
#pragma unroll
            for (int k = 0; k < VW; ++k) acc[v][k] = fma(coef[0], y0[k], fma(coef[RW - 1], y1[k], acc[v][k]));
          }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8 * slot);
    }
  }
  __syncthreads();   // every stage consumed: the ring is free for the reduction
  const int width = p.nv * VW;
  T* red = reinterpret_cast<T*>(bulk_smem);
  if (warp < CW) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      const int idx = lane + 32 * v;
      if (idx < p.nv) {
        for (int k = 0; k < VW; ++k) red[warp * width + idx * VW + k] = acc[v][k];
      }
    }
    if (MODE == PM_LSQR) {
      if constexpr (WIDE) sqacc = warp_sum(fma(qkeep, qkeep, sqacc));
      if (lane == 0) sqred[warp] = (double)sqacc;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < p.n; c += blockDim.x) {
    T s = 0;
#pragma unroll
    for (int w = 0; w < CW; ++w) s += red[w * width + c];
    p.Pblk[(int64_t)blockIdx.x * p.n + c] = s;
  }
  if (MODE == PM_LSQR && threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < CW; ++w) s += sqred[w];
    if constexpr (SCALED) {
      const double iqs = (double)__uint_as_float((254u << 23) - __float_as_uint(qs));   // 1 / qs
      s = s * iqs * iqs;
    }
    p.sq[blockIdx.x] = s;
  }
}

int bulk_blocks(int num_sms) { return num_sms; }

template <typename T, int VW, int MODE, bool SCALED = false>
static cudaError_t dispatch_bulk(BulkArgs<T> p, int nblk, int num_sms_unused, cudaStream_t st) {
  const int vpl = (p.nv + 31) / 32;
  const size_t stage_bytes = (size_t)kBulkRows * p.lda * sizeof(T);
  const size_t budget = 200 * 1024;
  int stages = (int)(budget / stage_bytes);
  if (stages > 12) stages = 12;
  if (stages < 2) return cudaErrorInvalidValue;
  p.stages = stages;
  p.rows_per_cta = ((p.m + nblk - 1) / nblk + kBulkRows - 1) / kBulkRows * kBulkRows;
  const size_t red_bytes = (size_t)kBulkRows * p.nv * VW * sizeof(T);
  size_t smem = (size_t)stages * stage_bytes;
  if (smem < red_bytes) smem = red_bytes;
  smem += 2 * stages * 8;
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_dyn_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<nblk, kBulkThreads<T>, smem, st>>>(p);
    return cudaGetLastError();
  };
  if (vpl <= 1) return go(pass_bulk_kernel<T, VW, 1, MODE, SCALED>);
  if (vpl <= 2) return go(pass_bulk_kernel<T, VW, 2, MODE, SCALED>);
  if (vpl <= 4) return go(pass_bulk_kernel<T, VW, 4, MODE, SCALED>);
  if (vpl <= 8) return go(pass_bulk_kernel<T, VW, 8, MODE, SCALED>);
  if constexpr (VW <= 2) {
    if (vpl <= 16) return go(pass_bulk_kernel<T, VW, 16, MODE, SCALED>);
  }
  return cudaErrorInvalidValue;
}

int pass_blocks(int num_sms) { return num_sms; }

template <typename T, int VW, int MODE>
static cudaError_t dispatch_pass(const PassArgs<T>& p, int nblk, cudaStream_t st) {
  const int vpl = (p.nv + 31) / 32;
  const size_t smem = (size_t)8 * p.nv * VW * sizeof(T);
  auto go = [&](auto kern) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e = allow_dyn_smem(kern, smem);
      if (e != cudaSuccess) return e;
    }
    kern<<<nblk, 256, smem, st>>>(p);
    return cudaGetLastError();
  };
  if (vpl <= 1) return go(pass_kernel<T, VW, 1, MODE>);
  if (vpl <= 2) return go(pass_kernel<T, VW, 2, MODE>);
  if (vpl <= 4) return go(pass_kernel<T, VW, 4, MODE>);
  if (vpl <= 8) return go(pass_kernel<T, VW, 8, MODE>);
  if constexpr (VW <= 2) {
    if (vpl <= 16) return go(pass_kernel<T, VW, 16, MODE>);
  }
  if constexpr (VW == 1) {
    if (vpl <= 32) return go(pass_kernel<T, VW, 32, MODE>);
  }
  return cudaErrorInvalidValue;
}

// Vector width for an FP64 matrix: double2 when rows and the base are 16-byte aligned.
static int f64_vw(const double* A, int64_t lda, int64_t n) {
  return ((reinterpret_cast<uintptr_t>(A) & 15) == 0 && (lda % 2) == 0 && (n % 2) == 0) ? 2 : 1;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// The bulk-streamed ring needs two stages of kBulkRows rows within its 200 KB of
// shared memory and a bulk instantiation for the row's vector count; wider rows
// (FP64 beyond 800 columns) take the register-blocked pass kernel instead.
template <typename T, int VW>
static bool bulk_fits(int64_t lda, int64_t nv) {
  const int64_t vpl = (nv + 31) / 32;
  return 2 * (size_t)kBulkRows * (size_t)lda * sizeof(T) <= (size_t)200 * 1024 &&
         (vpl <= 8 || (VW <= 2 && vpl <= 16));
}

template <typename T>
cudaError_t launch_pass_lsqr_t(const T* A, int64_t lda, int64_t m, int64_t n, const T* t,
                               const T* u_in, const double* cu_ptr, double cu_mul, T* u_out, T* Pblk,
                               double* sq, int nblk, const int* done, cudaStream_t st,
                               const double* sq_ref) {
  int vw = 4;
  bool bulk = aligned16(A);
  if constexpr (sizeof(T) == 4) {
    bulk = bulk && bulk_fits<float, 4>(lda, (lda + 3) / 4);
  } else {
    vw = f64_vw(A, lda, n);
    bulk = bulk && lda % 2 == 0 &&
           (vw == 2 ? bulk_fits<double, 2>(lda, n / 2) : bulk_fits<double, 1>(lda, n));
  }
  if (bulk) {
    BulkArgs<T> b{};
    b.A = A; b.lda = lda; b.m = m; b.n = (int)n;
    b.x = t; b.uin = u_in; b.uout = u_out; b.cu_ptr = cu_ptr; b.cu_mul = cu_mul;
    b.Pblk = Pblk; b.sq = sq; b.done = done; b.sq_ref = sq_ref;
    if constexpr (sizeof(T) == 4) {
      b.nv = (int)((lda + 3) / 4);
      if (sq_ref) return dispatch_bulk<float, 4, PM_LSQR, true>(b, nblk, 0, st);
      return dispatch_bulk<float, 4, PM_LSQR>(b, nblk, 0, st);
    } else {
      if (vw == 2) {
        b.nv = (int)(n / 2);
        return dispatch_bulk<double, 2, PM_LSQR>(b, nblk, 0, st);
      }
      b.nv = (int)n;
      return dispatch_bulk<double, 1, PM_LSQR>(b, nblk, 0, st);
    }
  }
  PassArgs<T> p{};
  p.A = A; p.lda = lda; p.m = m; p.n = (int)n;
  p.x = t; p.uin = u_in; p.uout = u_out; p.cu_ptr = cu_ptr; p.cu_mul = cu_mul;
  p.Pblk = Pblk; p.sq = sq; p.done = done;
  if constexpr (sizeof(T) == 4) {
    p.nv = (int)((lda + 3) / 4);   // A32 rows are zero padded to lda (a multiple of 4)
    return dispatch_pass<float, 4, PM_LSQR>(p, nblk, st);
  } else {
    if (vw == 2) {
      p.nv = (int)(n / 2);
      return dispatch_pass<double, 2, PM_LSQR>(p, nblk, st);
    }
    p.nv = (int)n;
    return dispatch_pass<double, 1, PM_LSQR>(p, nblk, st);
  }
}


template <typename TA>
cudaError_t launch_pass_fgm(const TA* A, int64_t lda, int64_t m, int64_t n, const TA* z,
                            const TA* v, TA* az, TA* Pblk, int nblk, const int* done, cudaStream_t st,
                            const int* jp, int64_t zs, int64_t vstr, int* err) {
  BulkArgs<TA> b{};
  b.A = A; b.lda = lda; b.m = m; b.n = (int)n;
  b.x = z; b.v = v; b.az = az; b.Pblk = Pblk; b.done = done; b.err = err;
  b.jp = jp; b.xstr = zs; b.vstr = vstr;
  if constexpr (sizeof(TA) == 4) {
    if (!aligned16(A) || (lda % 4) != 0) return cudaErrorInvalidValue;
    b.nv = (int)((lda + 3) / 4);
    return dispatch_bulk<float, 4, PM_FGM>(b, nblk, 0, st);
  } else {
    const int vw = f64_vw(A, lda, n);
    if (aligned16(A) && (lda % 2) == 0 &&
        (vw == 2 ? bulk_fits<double, 2>(lda, n / 2) : bulk_fits<double, 1>(lda, n))) {
      if (vw == 2) {
        b.nv = (int)(n / 2);
        return dispatch_bulk<double, 2, PM_FGM>(b, nblk, 0, st);
      }
      b.nv = (int)n;
      return dispatch_bulk<double, 1, PM_FGM>(b, nblk, 0, st);
    }
    PassArgs<double> q{};
    q.A = A; q.lda = lda; q.m = m; q.n = (int)n;
    q.x = z; q.v = v; q.az = az; q.Pblk = Pblk; q.done = done;
    q.jp = jp; q.xstr = zs; q.vstr = vstr;
    if (vw == 2) {
      q.nv = (int)(n / 2);
      return dispatch_pass<double, 2, PM_FGM>(q, nblk, st);
    }
    q.nv = (int)n;
    return dispatch_pass<double, 1, PM_FGM>(q, nblk, st);
  }
}
template cudaError_t launch_pass_fgm<float>(const float*, int64_t, int64_t, int64_t, const float*,
                                            const float*, float*, float*, int, const int*,
                                            cudaStream_t, const int*, int64_t, int64_t, int*);
template cudaError_t launch_pass_fgm<double>(const double*, int64_t, int64_t, int64_t, const double*,
                                             const double*, double*, double*, int, const int*,
                                             cudaStream_t, const int*, int64_t, int64_t, int*);

cudaError_t launch_pass_res(const double* A, int64_t lda, int64_t m, int64_t n, const double* x,
                            const double* r, const double* b, double* f, double* Pblk, int nblk,
                            cudaStream_t st) {
  const int vw = f64_vw(A, lda, n);
  if (aligned16(A) && lda % 2 == 0 &&
      (vw == 2 ? bulk_fits<double, 2>(lda, n / 2) : bulk_fits<double, 1>(lda, n))) {
    BulkArgs<double> q{};
    q.A = A; q.lda = lda; q.m = m; q.n = (int)n;
    q.x = x; q.r = r; q.b = b; q.f = f; q.Pblk = Pblk;
    if (f64_vw(A, lda, n) == 2) {
      q.nv = (int)(n / 2);
      return dispatch_bulk<double, 2, PM_RES>(q, nblk, 0, st);
    }
    q.nv = (int)n;
    return dispatch_bulk<double, 1, PM_RES>(q, nblk, 0, st);
  }
  PassArgs<double> p{};
  p.A = A; p.lda = lda; p.m = m; p.n = (int)n;
  p.x = x; p.r = r; p.b = b; p.f = f; p.Pblk = Pblk;
  if (f64_vw(A, lda, n) == 2) {
    p.nv = (int)(n / 2);
    return dispatch_pass<double, 2, PM_RES>(p, nblk, st);
  }
  p.nv = (int)n;
  return dispatch_pass<double, 1, PM_RES>(p, nblk, st);
}

// ------------------------------------------------------------ column sums
// A warp per column, lanes over the CTAs' partials, eight columns a CTA (32-byte pieces of
// the rows of P).  FP64 additions and FP32 -> FP64 conversions are what it costs (an SM
// does two a clock), so the columns are spread over many CTAs: 32 columns a CTA with a serial
// sum of 32 shares took 7 us at n = 500, 5 now.
template <typename TP>
__device__ __forceinline__ double colsum_warp(const TP* __restrict__ P, int nblk, int64_t n, int64_t c) {
  const int lane = threadIdx.x & 31;
  double s0 = 0.0, s1 = 0.0;
  int b = lane;
  for (; b + 32 < nblk; b += 64) {
    const TP p0 = P[(int64_t)b * n + c], p1 = P[(int64_t)(b + 32) * n + c];
    s0 += (double)p0;
    s1 += (double)p1;
  }
  if (b < nblk) s0 += (double)P[(int64_t)b * n + c];
  return warp_sum(s0 + s1);
}

template <typename TP, typename TO>
__device__ __forceinline__ void colsum_body(const TP* __restrict__ P, int nblk, int64_t n, const double* scale_ptr,
                                            double scale_mul, TO* __restrict__ out, const int* done, int64_t bx) {
  if (done && *done) return;
  const int64_t c = bx * kColsumCols + (threadIdx.x >> 5);
  if (c >= n) return;
  const double t = colsum_warp<TP>(P, nblk, n, c);
  if ((threadIdx.x & 31) == 0) out[c] = (TO)(t * ((scale_ptr ? *scale_ptr : 1.0) * scale_mul));
}

template <typename TP, typename TO>
__global__ void __launch_bounds__(kColsumCols * 32)
    colsum_kernel(const TP* __restrict__ P, int nblk, int64_t n, const double* scale_ptr,
                  double scale_mul, TO* __restrict__ out, const int* done) {
  colsum_body<TP, TO>(P, nblk, n, scale_ptr, scale_mul, out, done, blockIdx.x);
}

template <typename TP, typename TO>
cudaError_t launch_colsum(const TP* P, int nblk, int64_t n, const double* scale_ptr, double scale_mul,
                          TO* out, const int* done, cudaStream_t st) {
  colsum_kernel<TP, TO><<<(unsigned)((n + kColsumCols - 1) / kColsumCols), kColsumCols * 32, 0, st>>>(
      P, nblk, n, scale_ptr, scale_mul, out, done);
  return cudaGetLastError();
}
template cudaError_t launch_colsum<float, float>(const float*, int, int64_t, const double*, double,
                                                 float*, const int*, cudaStream_t);
template cudaError_t launch_colsum<double, double>(const double*, int, int64_t, const double*, double,
                                                   double*, const int*, cudaStream_t);
template cudaError_t launch_colsum<double, float>(const double*, int, int64_t, const double*, double,
                                                  float*, const int*, cudaStream_t);
template cudaError_t launch_colsum<float, double>(const float*, int, int64_t, const double*, double,
                                                  double*, const int*, cudaStream_t);

// ============================================================ LSQR kernels
template <typename TP>
cudaError_t launch_pass_lsqr_any(const TP* A, int64_t lda, int64_t m, int64_t n, const TP* t,
                                 const TP* u_in, const double* cu_ptr, double cu_mul, TP* u_out,
                                 TP* Pblk, double* sq, int nblk, const int* done, cudaStream_t st,
                                 const double* sq_ref) {
  return launch_pass_lsqr_t<TP>(A, lda, m, n, t, u_in, cu_ptr, cu_mul, u_out, Pblk, sq, nblk, done, st, sq_ref);
}
template cudaError_t launch_pass_lsqr_any<float>(const float*, int64_t, int64_t, int64_t, const float*,
                                                 const float*, const double*, double, float*, float*,
                                                 double*, int, const int*, cudaStream_t, const double*);
template cudaError_t launch_pass_lsqr_any<double>(const double*, int64_t, int64_t, int64_t, const double*,
                                                  const double*, const double*, double, double*,
                                                  double*, double*, int, const int*, cudaStream_t,
                                                  const double*);

// ------------------------------------------------------------ fused LSQR step
// beta = ||q|| from the per-CTA sums of squares (every CTA recomputes it);
// out[c] = (A^T q)_c / beta.  Block 0 publishes beta and 1/beta.
template <typename TP>
__device__ __forceinline__ void lsqr_colsum_body(const TP* __restrict__ P, int nblk, int64_t n, const double* sq,
                                                 LsqrState* st, bool init, TP* __restrict__ out, int64_t bx) {
  if (!init && st->done) return;
  __shared__ double us_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == kColsumCols) {   // a warp of its own: beta, its square root and reciprocal once
    double q = 0.0;
    for (int b = lane; b < nblk; b += 32) q += sq[b];
    q = warp_sum(q);
    if (lane == 0) {
      const double beta = sqrt(q);
      const double us = beta > 0.0 ? 1.0 / beta : 0.0;
      us_s = us;
      if (bx == 0) {
        st->beta = beta;
        st->us = us;
        if (init) st->phibar = beta;
      }
    }
  }
  const int64_t c = bx * kColsumCols + warp;
  double t = 0.0;
  if (warp < kColsumCols && c < n) t = colsum_warp<TP>(P, nblk, n, c);
  __syncthreads();
  if (warp < kColsumCols && c < n && lane == 0) out[c] = (TP)(t * us_s);
}

template <typename TP>
__global__ void __launch_bounds__((kColsumCols + 1) * 32)
    lsqr_colsum_kernel(const TP* __restrict__ P, int nblk, int64_t n, const double* sq,
                       LsqrState* st, bool init, TP* __restrict__ out) {
  lsqr_colsum_body<TP>(P, nblk, n, sq, st, init, out, blockIdx.x);
}

// The plane rotation and the stopping tests of one step, by one warp: square roots and
// quotients that do not depend on one another run in different lanes (each is a chain of some
// 40 FP64 operations).  coef (shared): the factors of the z and w updates.
__device__ __forceinline__ void lsqr_scalars(LsqrState* st, bool init, double alpha, double beta, double* coef) {
  const int lane = threadIdx.x & 31;
  if (init) {
    if (lane == 0) {
      st->alpha = alpha;
      st->rhobar = alpha;
      st->anorm2 = 0.0;
      st->its = 0;
      st->normr = beta;
      st->normar = alpha * beta;
      st->normA = 0.0;
      st->flag = (beta == 0.0 || alpha == 0.0) ? 3 : 0;
      st->done = (st->flag != 0 || st->maxit <= 0) ? 1 : 0;
      coef[0] = 0.0;
      coef[1] = 0.0;
      st->cu = -alpha * st->us;
    }
    return;
  }
  const double alpha_old = st->alpha, rhobar = st->rhobar, phibar0 = st->phibar;
  const double anorm2 = st->anorm2 + alpha_old * alpha_old + beta * beta;
  const double root = sqrt(lane == 0 ? rhobar * rhobar + beta * beta : anorm2);
  const double rho = __shfl_sync(0xffffffffu, root, 0), normA = __shfl_sync(0xffffffffu, root, 1);
  const double q1 = (lane == 0 ? rhobar : beta) / rho;
  const double c = __shfl_sync(0xffffffffu, q1, 0), sn = __shfl_sync(0xffffffffu, q1, 1);
  const double theta = sn * alpha, phi = c * phibar0, phibar = sn * phibar0;
  const double q2 = (lane == 0 ? phi : theta) / rho;
  if (lane < 2) coef[lane] = q2;
  if (lane == 0) {
    st->rhobar = -c * alpha;
    st->phibar = phibar;
    st->anorm2 = anorm2;
    st->alpha = alpha;
    st->its += 1;
    st->normr = fabs(phibar);
    st->normar = fabs(phibar * alpha * c);
    st->normA = normA;
    int flag = 0;
    if (st->normr <= st->tol * st->normb) flag = 1;
    else if (st->normar <= st->tol * normA * st->normr) flag = 2;
    else if (beta == 0.0 || alpha == 0.0) flag = 3;
    st->flag = flag;
    st->done = (flag != 0 || st->its >= st->maxit) ? 1 : 0;
    st->cu = -alpha * st->us;
  }
}

// One CTA: vt = R^-T s ; (init) alpha v = vt, w = v, z = 0 ; (iteration)
// alpha v = vt - beta v, plane rotation, z += (phi/rho) w, w = v - (theta/rho) w,
// stopping tests ; then t = R^-1 v for the next pass.
template <typename T>
__device__ __forceinline__ void lsqr_step_body(const Tri<T>& f, const T* __restrict__ s, T* __restrict__ v,
                                               T* __restrict__ w, T* __restrict__ z, T* __restrict__ t,
                                               LsqrState* st, bool init) {
  if (!init && st->done) return;
  __shared__ T xs[1024];
  __shared__ double red[33];
  __shared__ double coef[3];
  extern __shared__ __align__(16) unsigned char step_buf[];
  const int n = (int)f.n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) xs[i] = s[i];
  __syncthreads();
  if (!block_trsv<T, false>(f.L, f.ld, f.DL, n, xs, step_buf, f.err)) return;   // xs = R^-T s
  const double beta = st->beta;
  double ss = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const T vv = init ? xs[i] : xs[i] - (T)beta * v[i];
    ss += (double)vv * (double)vv;
  }
  ss = block_sum_d(ss, red);
  if (threadIdx.x < 32) {   // one warp: the FP64 roots and quotients
    const double alpha = sqrt(ss);
    lsqr_scalars(st, init, alpha, beta, coef);
    if (threadIdx.x == 0) coef[2] = alpha > 0.0 ? 1.0 / alpha : 0.0;
  }
  __syncthreads();
  const T ia = (T)coef[2];
  const T c0 = (T)coef[0], c1 = (T)coef[1];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const T vn = (init ? xs[i] : xs[i] - (T)beta * v[i]) * ia;
    if (init) {
      w[i] = vn;
      z[i] = T(0);
    } else {
      const T wi = w[i];
      z[i] = z[i] + c0 * wi;
      w[i] = vn - c1 * wi;
    }
    v[i] = vn;
    xs[i] = vn;
  }
  __syncthreads();
  if (!block_trsv<T, true>(f.R, f.ld, f.DU, n, xs, step_buf, f.err)) return;    // t = R^-1 v
  for (int i = threadIdx.x; i < n; i += blockDim.x) t[i] = xs[i];
}

// The step of one problem by two launches over the rows of X = R^-1 (a warp per row):
//   1: vv = X^T s - beta v (init: X^T s), and the CTA's sum of squares;
//   2: alpha = ||vv||; t = X (vv / alpha) for the next pass; CTA 0 also does the scalars and the
//      vectors v, w, z.  (A CTA that starts after CTA 0 has set done skips its rows of t: no
//      pass reads them then.)
// On one CTA with two triangular solves the step took 20 us at n = 50 and 46 us at n = 500.
// Accuracy: k_trsv.cu (trinv_kernel).  FP64 solves (tol 1e-14), median error of eight problems of m = 2000, n = 50
// / m = 6000, n = 180 against extended precision, substituting: kappa 1e3 1.6e-15 / 2.2e-15, 1e6 9.4e-11 / 6.7e-11, 1e9
// 1.5e-8 / 3.3e-9; now (with q^2 summed in FP64 too): 1.8e-15 / 2.0e-15, 3.0e-11 / 4.0e-11, 3.0e-9 / 1.9e-9.
template <typename T>
__global__ void __launch_bounds__(kTrimvWarps * 32)
    lsqr_step1_kernel(const T* __restrict__ XT, int64_t ld, int n, const T* __restrict__ s, const T* __restrict__ v,
                      T* __restrict__ vv, double* __restrict__ part, const LsqrState* st, bool init) {
  if (!init && st->done) return;
  __shared__ __align__(16) T ysm[1024];
  __shared__ double sq[kTrimvWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * kTrimvWarps + warp;
  const int c1 = min((int)ld, (int)(blockIdx.x + 1) * kTrimvWarps + 4);
  for (int i = threadIdx.x; i < c1; i += blockDim.x) ysm[i] = i < n ? s[i] : T(0);
  __syncthreads();
  if (r < n) {
    T x = trimv_row<T, true>(XT + (size_t)r * ld, r, n, ysm);
    if (!init) x -= (T)st->beta * v[r];
    if (lane == 0) {
      vv[r] = x;
      sq[warp] = (double)x * (double)x;
    }
  } else if (lane == 0) {
    sq[warp] = 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double q = 0.0;
#pragma unroll
    for (int w = 0; w < kTrimvWarps; ++w) q += sq[w];
    part[blockIdx.x] = q;
  }
}

template <typename T>
__global__ void __launch_bounds__(kTrimvWarps * 32)
    lsqr_step2_kernel(const T* __restrict__ X, int64_t ld, int n, const T* __restrict__ vv,
                      const double* __restrict__ part, T* __restrict__ v, T* __restrict__ w, T* __restrict__ z,
                      T* __restrict__ t, LsqrState* st, bool init) {
  if (!init && st->done) return;
  __shared__ __align__(16) T ysm[1024];
  __shared__ double coef[2], alpha_s;
  __shared__ T ia_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {   // once: an FP64 root and quotient in every warp would cost microseconds
    double q = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) q += part[b];
    const double al = sqrt(warp_sum(q));
    if (lane == 0) {
      alpha_s = al;
      ia_s = al > 0.0 ? (T)(1.0 / al) : T(0);
    }
  }
  __syncthreads();
  const double alpha = alpha_s;
  const T ia = ia_s;
  const int c0 = (blockIdx.x * kTrimvWarps / 4) * 4;
  for (int i = c0 + threadIdx.x; i < (int)ld; i += blockDim.x) ysm[i] = i < n ? vv[i] * ia : T(0);
  __syncthreads();
  const int r = blockIdx.x * kTrimvWarps + warp;
  if (r < n) {
    const T x = trimv_row<T, false>(X + (size_t)r * ld, r, n, ysm);
    if (lane == 0) t[r] = x;
  }
  if (blockIdx.x == 0) {   // ysm holds all of v here
    if (warp == 0) lsqr_scalars(st, init, alpha, st->beta, coef);
    __syncthreads();
    const T f0 = (T)coef[0], f1 = (T)coef[1];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const T vn = ysm[i];
      if (init) {
        w[i] = vn;
        z[i] = T(0);
      } else {
        const T wi = w[i];
        z[i] = z[i] + f0 * wi;
        w[i] = vn - f1 * wi;
      }
      v[i] = vn;
    }
  }
}

// The step on one CTA with two substitutions, for a solve of a single iteration.
__global__ void __launch_bounds__(kTrsvThreads)
    lsqr_step_kernel(const Tri<float> f, const float* __restrict__ s, float* __restrict__ v, float* __restrict__ w,
                     float* __restrict__ z, float* __restrict__ t, LsqrState* st, bool init) {
  lsqr_step_body<float>(f, s, v, w, z, t, st, init);
}

template <typename T>
cudaError_t launch_lsqr_colsum(const T* P, int nblk, int64_t n, const double* sq, LsqrState* st,
                               bool init, T* out, cudaStream_t s) {
  lsqr_colsum_kernel<T><<<(unsigned)((n + kColsumCols - 1) / kColsumCols), (kColsumCols + 1) * 32, 0, s>>>(P, nblk, n, sq, st,
                                                                                                      init, out);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_lsqr_step(const Tri<T>& f, const T* s, T* v, T* w, T* z, T* t, T* vv, double* part,
                             LsqrState* st, bool init, cudaStream_t strm) {
  if (f.n > 1024) return cudaErrorInvalidValue;
  if (!f.X || !f.XT) {
    if constexpr (sizeof(T) == 4) {
      const size_t smem = TrsvSmem<T>::bytes;
      cudaError_t e = allow_dyn_smem(lsqr_step_kernel, smem);
      if (e != cudaSuccess) return e;
      lsqr_step_kernel<<<1, kTrsvThreads, smem, strm>>>(f, s, v, w, z, t, st, init);
      return cudaGetLastError();
    } else {
      return cudaErrorInvalidValue;
    }
  }
  const unsigned grid = (unsigned)((f.n + kTrimvWarps - 1) / kTrimvWarps);
  lsqr_step1_kernel<T><<<grid, kTrimvWarps * 32, 0, strm>>>(f.XT, f.ld, (int)f.n, s, v, vv, part, st, init);
  lsqr_step2_kernel<T><<<grid, kTrimvWarps * 32, 0, strm>>>(f.X, f.ld, (int)f.n, vv, part, v, w, z, t, st, init);
  return cudaGetLastError();
}
template cudaError_t launch_lsqr_colsum<float>(const float*, int, int64_t, const double*, LsqrState*, bool, float*, cudaStream_t);
template cudaError_t launch_lsqr_colsum<double>(const double*, int, int64_t, const double*, LsqrState*, bool, double*, cudaStream_t);
template cudaError_t launch_lsqr_step<float>(const Tri<float>&, const float*, float*, float*, float*, float*, float*, double*, LsqrState*, bool, cudaStream_t);
template cudaError_t launch_lsqr_step<double>(const Tri<double>&, const double*, double*, double*, double*, double*, double*, double*, LsqrState*, bool, cudaStream_t);

// ============================================================ vector kernels
// out[i] = x[i] * a + y[i] * b  (types converted), i < len
template <typename TX, typename TY, typename TO>
__global__ void axpby_kernel(const TX* x, double a, const TY* y, double b, TO* out, int64_t len) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= len) return;
  double v = (double)x[i] * a;
  if (y) v += (double)y[i] * b;
  out[i] = (TO)v;
}

template <typename TX, typename TY, typename TO>
cudaError_t launch_axpby(const TX* x, double a, const TY* y, double b, TO* out, int64_t len,
                         cudaStream_t st) {
  if (len <= 0) return cudaSuccess;
  axpby_kernel<TX, TY, TO><<<(unsigned)((len + 255) / 256), 256, 0, st>>>(x, a, y, b, out, len);
  return cudaGetLastError();
}
template cudaError_t launch_axpby<double, double, float>(const double*, double, const double*, double, float*, int64_t, cudaStream_t);
template cudaError_t launch_axpby<double, double, double>(const double*, double, const double*, double, double*, int64_t, cudaStream_t);
template cudaError_t launch_axpby<float, double, double>(const float*, double, const double*, double, double*, int64_t, cudaStream_t);
template cudaError_t launch_axpby<double, float, double>(const double*, double, const float*, double, double*, int64_t, cudaStream_t);
template cudaError_t launch_axpby<float, float, double>(const float*, double, const float*, double, double*, int64_t, cudaStream_t);
template cudaError_t launch_axpby<float, float, float>(const float*, double, const float*, double, float*, int64_t, cudaStream_t);

// partial[b] = sum over the block's range of x_i * y_i (x, y double; y = x for norms)
__global__ void dot_partial_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                   int64_t len, double* partial) {
  __shared__ double red[33];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x)
    s += x[i] * y[i];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void sum_partials_kernel(const double* partial, int nblk, double* out, bool take_sqrt) {
  __shared__ double red[33];
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += partial[b];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) *out = take_sqrt ? sqrt(s) : s;
}

cudaError_t launch_dot(const double* x, const double* y, int64_t len, double* partial, int nblk,
                       double* out, bool take_sqrt, cudaStream_t st) {
  dot_partial_kernel<<<nblk, 256, 0, st>>>(x, y, len, partial);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  sum_partials_kernel<<<1, 1024, 0, st>>>(partial, nblk, out, take_sqrt);
  return cudaGetLastError();
}

// ============================================================ FGMRES kernels
// V column-major with leading dimension ld = m + n; H column-major (maxit+1 rows).
__global__ void gm_init_kernel(const double* sq_partial, int nblk, GmState* st, double* g) {
  __shared__ double red[33];
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += sq_partial[b];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) {
    const double beta = sqrt(s);
    st->beta0 = beta;
    st->inv_h = beta > 0.0 ? 1.0 / beta : 0.0;
    st->j = 0;
    st->relres = beta > 0.0 ? 1.0 : 0.0;
    st->done = (beta == 0.0 || st->maxit <= 0) ? 1 : 0;
    g[0] = beta;
  }
}

// h_{j+1,j} = sqrt(s); Givens rotations on column j; residual estimate; j++.
// One warp (warp 0 of block 0 of the Arnoldi step), with the unrotated column h_{0..j, j}
// in shared memory (hcol, rotated in place): the other warps of the block keep working.
// The rotations carry p_{i+1} = -s_i p_i + c_i h_{i+1} down the column: a linear recurrence,
// taken as a scan of affine maps over the lanes (four rotations a lane at most), and the
// square roots and quotients that do not depend on one another run in different lanes.
// (As one serial chain of FP64 operations with hypot it took about 9 us at j = 25; 3 us now.)
// pre (shared): cs[0..j), sn[0..j) at pre + 128, then g_j, beta0 and tol,
// loaded by gm_finish_prefetch earlier in the kernel.
__device__ __forceinline__ void gm_finish_prefetch(const GmState* st, const double* cs, const double* sn,
                                                   const double* g, double* pre) {
  const int j = st->j;
  for (int i = threadIdx.x; i < j; i += blockDim.x) {
    pre[i] = cs[i];
    pre[128 + i] = sn[i];
  }
  if (threadIdx.x == 0) {
    pre[256] = g[j];
    pre[257] = st->beta0;
    pre[258] = st->tol;
  }
}
__device__ void gm_finish_warp(double s, int j, const double* pre, GmState* st, double* hcol, double* H, int ldh,
                               double* cs, double* sn, double* g) {
  const int lane = threadIdx.x & 31;
  const int per = (j + 31) >> 5;   // rotations of a lane
  const int i0 = min(j, lane * per), i1 = min(j, i0 + per);
  double c4[4], s4[4], h4[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (i0 + q < i1) {
      c4[q] = pre[i0 + q];
      s4[q] = pre[128 + i0 + q];
      h4[q] = hcol[i0 + q + 1];
    }
  const double h0 = hcol[0];
  double A = 1.0, B = 0.0;   // p after the lane's rotations = A p + B
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (i0 + q < i1) {
      B = fma(-s4[q], B, c4[q] * h4[q]);
      A *= -s4[q];
    }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double Al = __shfl_up_sync(0xffffffffu, A, o), Bl = __shfl_up_sync(0xffffffffu, B, o);
    if (lane >= o) {
      B = fma(A, Bl, B);
      A *= Al;
    }
  }
  const double pend = fma(A, h0, B);   // p after this lane's rotations
  double p = __shfl_up_sync(0xffffffffu, pend, 1);
  if (lane == 0) p = h0;
  const double hj = __shfl_sync(0xffffffffu, pend, 31);   // the rotated h_j
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (i0 + q < i1) {
      hcol[i0 + q] = fma(c4[q], p, s4[q] * h4[q]);
      p = fma(-s4[q], p, c4[q] * h4[q]);
    }
  // lane 0: h_{j+1,j}; lane 1: the rotated diagonal sqrt(h_j^2 + h_{j+1,j}^2)
  const double root = sqrt(lane == 0 ? s : fma(hj, hj, s));
  const double hn = __shfl_sync(0xffffffffu, root, 0);
  double den = __shfl_sync(0xffffffffu, root, 1);
  if (__double2hiint(den) < 0x20C00000) den = hypot(hj, hn);   // below about 1e-150: the squares' range (integer test)
  const double gj = pre[256];
  // lane 0: 1 / h_{j+1,j}; lanes 1, 2: the rotation; lane 3: |g_j| / beta0
  const double num = lane == 0 ? 1.0 : lane == 1 ? hj : lane == 2 ? hn : fabs(gj);
  const double dv = lane == 0 ? hn : lane == 3 ? pre[257] : den;
  // positive numbers are tested and compared by their bits (an FP64 comparison takes the pipe)
  const double qt = __double_as_longlong(dv) > 0 ? num / dv : (lane == 1 ? 1.0 : 0.0);
  const double cj = __shfl_sync(0xffffffffu, qt, 1), sj = __shfl_sync(0xffffffffu, qt, 2);
  const double rel = fabs(sj) * __shfl_sync(0xffffffffu, qt, 3);
  if (lane == 0) {
    cs[j] = cj;
    sn[j] = sj;
    hcol[j] = den;
    hcol[j + 1] = 0.0;
    g[j + 1] = -sj * gj;
    g[j] = cj * gj;
    st->relres = rel;
    st->inv_h = qt;
    st->j = j + 1;
    st->done = (__double_as_longlong(rel) <= __double_as_longlong(pre[258]) || j + 1 >= st->maxit ||
                __double_as_longlong(hn) == 0) ? 1 : 0;
  }
  __syncwarp();
  double* hc = H + (int64_t)j * ldh;
  for (int i = lane; i <= j + 1; i += 32) hc[i] = hcol[i];
}

// ---------------------------------------------------------------- fused Arnoldi step
// One launch per FGMRES iteration, 512-thread CTAs, each owning a contiguous row range of
// the length-(m+n) vectors; FP64 throughout.  The CTA's rows of w and of as many basis
// columns as fit live in shared memory (staged once with asynchronous copies): the up to four
// sweeps of a step then wait for no L2 loads.  Short vectors (SUMS = 1, up to kGmClusterRows
// rows) run on one cluster of sixteen CTAs that add their partials through distributed shared
// memory; the others (SUMS = 0) as a cooperative launch of at most one CTA per SM and 64 rows.
//   w_top = v_top + A z; partials of h = V^T w and of ||w||^2 (eight basis columns per
//   sweep over the rows, so w is read once per eight columns)
//   [sum 1 over the CTAs]
//   Kahan's "twice is enough": the first pass loses more than half of ||w||^2 iff
//   ||h||^2 > ||w||^2 / 2 (Pythagoras, decided before the update).  Otherwise
//   ||w - V h||^2 = ||w||^2 - ||h||^2 within a few units of FP64 rounding (V orthonormal
//   to working accuracy, no cancellation below one half), so the update writes the new
//   column v_{j+1} = (w - V h) / h_{j+1,j} directly: one sum per step.
//   With the second pass: w1 = w - V h; partials of h2 = V^T w1 and ||w1||^2 [sum 2];
//   v_{j+1} = (w1 - V h2) / sqrt(||w1||^2 - ||h2||^2) (h2 is of rounding size).
//   The last CTA adds h (and h2) to the Hessenberg column and applies the Givens rotations.
// Bound by FP64 (two FMAs a clock an SM) and by the sums (about 3 us each over the grid, under
// 1 us in a cluster): sums are arranged for few FP64 operations (one CTA per column in the
// grid sum, warp_reduce8 in the partials, one warp for ||h||^2, roots and quotients).  With w
// and V read from L2 in every sweep, sums by the last CTA to arrive and the Givens rotations as
// one serial chain, j = 25 on average: 40 -> 19 us at m = 1000, n = 100 and 51 -> 36 us at m = 1e5,
// n = 500, where the four sweeps of a step with the second pass are 17 us of FMAs.
// The syncs wait with a bounded spin; an expired wait records DEV_TIMEOUT_GRID and the
// kernel returns.
constexpr int kGmThreads = 512;
constexpr int kGmGroup = 8;   // basis columns per sweep of the partial dot products
template <typename TAZ>
struct GmStepArgs {
  double* V;
  int64_t ld, len, m;
  double* w;
  const TAZ* az;
  GmState* st;
  int maxc, ldh;
  double* Dp;     // [maxc + 1][ldd] partials, one column per block (row ncols: the squared norm)
  double* hsum;   // [maxc + 1] column sums
  double* H;
  double* cs;
  double* sn;
  double* g;
  float* v32;
  int* err;
  int ldd;        // leading dimension of Dp (>= the grid size)
  uint64_t wait_ns;   // limit of each grid-sync wait
  double alpha;       // w_top = alpha v_top + A z (Sec. 4.1 scaling; 1 unscaled)
  unsigned long long* seq;   // arrival counter of the grid syncs (zero before the solve)
  int expire;         // wait for one arrival more than the grid makes (the timeout test)
  int slab;           // basis columns that fit in the dynamic shared memory beside w
};

// Dp[c][block] = sum over rows [r0, r1) of V[c][i] w[i] for c < ncols; Dp[ncols][block] = sum of w[i]^2.
// The (ncols + 1) sums form G groups of eight; the CTA's rows are cut into S slices with
// G x S close to the warp count, and each warp takes one (group, slice) task: its lanes
// stride over the slice two rows at a time (18 loads in flight), one butterfly reduces
// the eight sums over the warp, and one thread per column adds the S slice sums in slice
// order.  Every partial is reduced once, whatever the number of rows per CTA.
constexpr int kGmRed = 160;   // doubles of the slice-sum buffer (>= max(16, G) x 8 with G <= 17);
constexpr int kGmRedWs = kGmRed + (512 / 32) * 32;   // with the warps' sums of the second form

// The eight sums of one task over rows [s0, s1) (V and w indexed by the row); lane L returns
// the warp total of sum (L >> 2) & 7.  A warp's FP64 instruction takes 16 cycles of the SM's one
// pipe whatever lanes are active, so the warp walks the rows together (zeros past s1).
__device__ __forceinline__ double gm_task(const double* __restrict__ V, int64_t ld, const double* __restrict__ w,
                                          int64_t s0, int64_t s1, int c0, int ncols) {
  const int lane = threadIdx.x & 31;
  double t[kGmGroup];
#pragma unroll
  for (int k = 0; k < kGmGroup; ++k) t[k] = 0.0;
  int64_t i = s0 + lane;
  if (c0 + kGmGroup <= ncols) {   // eight basis columns, no norm
    int64_t rows = s1 - s0;
    for (; rows >= 64; rows -= 64, i += 64) {
      const double wa = w[i], wb = w[i + 32];
      double va[kGmGroup], vb[kGmGroup];
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k) {
        va[k] = V[(int64_t)(c0 + k) * ld + i];
        vb[k] = V[(int64_t)(c0 + k) * ld + i + 32];
      }
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k) t[k] = fma(vb[k], wb, fma(va[k], wa, t[k]));
    }
    for (; rows > 0; rows -= 32, i += 32) {
      const bool in = i < s1;
      const double wa = in ? w[i] : 0.0;
      double va[kGmGroup];
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k) va[k] = in ? V[(int64_t)(c0 + k) * ld + i] : 0.0;
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k) t[k] = fma(va[k], wa, t[k]);
    }
  } else {
    for (int64_t rows = s1 - s0; rows > 0; rows -= 32, i += 32) {
      const bool in = i < s1;
      const double wi = in ? w[i] : 0.0;
      double v[kGmGroup];
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k)
        v[k] = c0 + k == ncols ? wi : (c0 + k < ncols && in ? V[(int64_t)(c0 + k) * ld + i] : 0.0);
#pragma unroll
      for (int k = 0; k < kGmGroup; ++k)
        if (c0 + k <= ncols) t[k] = fma(v[k], wi, t[k]);
    }
  }
  static_assert(kGmGroup == 8, "warp_reduce8 reduces eight sums");
  return warp_reduce8(t);
}

// Partials of V^T w and ||w||^2 over the CTA's rows [r0, r1) into Dp[c * ldd + blk], c <= ncols.
// nfit: the first nfit columns (a multiple of eight, or all) are also in shared memory, row i
// of column c at Vs[c * vld + i] (vld odd).  Two forms, by the FP64 instructions they take:
//  * lanes over rows, a warp per (group of eight sums, slice of rows), a nine-addition
//    reduction per task;
//  * lanes over the sums (all columns in shared memory, at most 32 sums): a row per
//    instruction -- two, four or eight where the sums leave lanes free -- and no reduction
//    but one addition per doubling and the sum over the warps.
__device__ __forceinline__ void gm_partials(const double* __restrict__ V, int64_t ld,
                                            const double* Vs, int64_t vld, int nfit,
                                            const double* __restrict__ w, int64_t r0, int64_t r1,
                                            int ncols, double* Dp, int ldd, double* red /* [kGmRed] */,
                                            int64_t blk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int G = (ncols + kGmGroup) / kGmGroup;   // groups covering ncols + 1 sums
  const int rows = (int)(r1 - r0);
  // slices of whole warp steps: enough tasks for eight warps (they saturate the pipe)
  // (more where V comes from global memory: loads in flight)
  const int S = max(1, min(min(nw / G, nfit > 0 ? (8 + G - 1) / G : nw), rows / 32));
  const int lp = ncols + 1 <= 4 ? 2 : ncols + 1 <= 8 ? 3 : ncols + 1 <= 16 ? 4 : 5;   // 2^lp lanes for the sums
  const int by_rows = ((rows + 31) / 32) * (ncols + 1) + 9 * G * S;
  const int by_sums = (rows >> (5 - lp)) + (5 - lp + 1) * nw;
  if (nfit >= ncols && ncols + 1 <= 32 && by_sums < by_rows) {
    const int c = lane & ((1 << lp) - 1), ph = lane >> lp, np = 32 >> lp;
    const double* vc = c < ncols ? Vs + (int64_t)c * vld : w;   // the last sum is w^T w
    double t = 0.0;
    const int64_t step = (int64_t)nw * np;
    int64_t i = r0 + (int64_t)warp * np;
    for (; i + 3 * step + np <= r1; i += 4 * step) {   // whole row groups, four in flight
      double v[4], x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[q] = vc[i + q * step + ph];
        x[q] = w[i + q * step + ph];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) t = fma(v[q], x[q], t);
    }
    for (; i < r1; i += step) {
      const bool in = i + ph < r1;
      const double v = in ? vc[i + ph] : 0.0, x = in ? w[i + ph] : 0.0;
      t = fma(v, x, t);
    }
    for (int o = 1 << lp; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    double* rw = red + kGmRed;   // [warps][32]
    rw[warp * 32 + lane] = t;
    __syncthreads();
    if (warp < 4) {   // four warps add a quarter of the warps each, one adds the quarters
      double s = rw[warp * 32 + lane];
      for (int k = warp + 4; k < nw; k += 4) s += rw[k * 32 + lane];
      rw[warp * 32 + lane] = s;
    }
    __syncthreads();
    if (warp == 0 && lane <= ncols)
      Dp[(int64_t)lane * ldd + blk] = (rw[lane] + rw[32 + lane]) + (rw[64 + lane] + rw[96 + lane]);
    __syncthreads();
    return;
  }
  const int64_t per = ((rows + S - 1) / S + 31) / 32 * 32;
  for (int task = warp; task < G * S; task += nw) {
    const int g = task % G, sl = task / G, c0 = g * kGmGroup;
    const int64_t s0 = min(r1, r0 + (int64_t)sl * per), s1 = min(r1, s0 + per);
    const double tot = (c0 + kGmGroup <= nfit || nfit >= ncols) ? gm_task(Vs, vld, w, s0, s1, c0, ncols)
                                                                : gm_task(V, ld, w, s0, s1, c0, ncols);
    if ((lane & 3) == 0) red[(sl * G + g) * kGmGroup + ((lane >> 2) & 7)] = tot;
  }
  __syncthreads();
  for (int c = threadIdx.x; c <= ncols; c += blockDim.x) {
    const int g = c / kGmGroup, k = c % kGmGroup;
    double s = red[g * kGmGroup + k];
    for (int sl = 1; sl < S; ++sl) s += red[(sl * G + g) * kGmGroup + k];
    Dp[(int64_t)c * ldd + blk] = s;   // column-major: [column][block]
  }
  __syncthreads();
}

// One grid-wide rendezvous on a 64-bit arrival counter: thread 0 of each CTA takes a ticket
// with a release add; the counter is zeroed before the solve and every launch of the solve has
// the same grid, so the tickets of one rendezvous fill [k nb, (k + 1) nb) and it is complete
// when the counter reaches (k + 1) nb.  Thread 0 waits for that (acquire loads, bounded;
// plus_one: for one more arrival, which never comes -- the timeout test).  Writes before it
// are visible to every thread of every CTA after it.  False if the wait ran out.
__device__ __forceinline__ unsigned long long atom_add_release_u64(unsigned long long* p, unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.add.release.gpu.global.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool gm_rendezvous(unsigned long long* ctr, int plus_one, int* err, uint64_t wait_ns) {
  int ok = 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned nb = gridDim.x;
    const unsigned long long ticket = atom_add_release_u64(ctr, 1ull);
    const unsigned long long target = (ticket / nb + 1ull) * nb + (plus_one ? 1ull : 0ull);
    if (ld_acquire_u64(ctr) < target) {
      const uint64_t t0 = globaltimer_ns();
      while (ld_acquire_u64(ctr) < target) {
        if (globaltimer_ns() - t0 > wait_ns) {
          set_error(err, DEV_TIMEOUT_GRID);
          ok = 0;
          break;
        }
      }
    }
  }
  return __syncthreads_and(ok) != 0;
}

// hs[c] = sum over the CTAs of Dp[c][.], c < cols, the same value in every CTA.  Few CTAs:
// every CTA adds the partials itself, a thread per column.  Many: CTA b adds columns b,
// b + nb, ... (a warp per column) and a second rendezvous publishes the sums in hsum (adding
// all of them in every CTA would cost 152 x 50 FP64 additions a CTA, in the last CTA to
// arrive the same serially).  Dp and hsum are not those of the step's other grid sum.
constexpr int kGmFewCtas = 32;
__device__ __forceinline__ bool gm_grid_sums(const double* Dp, int ldd, double* hsum, int cols,
                                             unsigned long long* ctr, int plus_one, int* err, uint64_t wait_ns,
                                             double* hs) {
  const int nb = (int)gridDim.x;
  if (!gm_rendezvous(ctr, plus_one, err, wait_ns)) return false;
  if (nb <= kGmFewCtas) {
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
      double s = 0.0;
      for (int q = 0; q < nb; ++q) s += __ldcg(Dp + (int64_t)c * ldd + q);
      hs[c] = s;
    }
  } else {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = (int)blockIdx.x + warp * nb;
    if (c < cols) {
      const double* col = Dp + (int64_t)c * ldd;
      double t0 = 0.0, t1 = 0.0;
      int q = lane;
      for (; q + 32 < nb; q += 64) {
        t0 += __ldcg(col + q);
        t1 += __ldcg(col + q + 32);
      }
      if (q < nb) t0 += __ldcg(col + q);
      const double s = warp_sum(t0 + t1);
      if (lane == 0) hsum[c] = s;
    }
    if (!gm_rendezvous(ctr, 0, err, wait_ns)) return false;
    for (int k = threadIdx.x; k < cols; k += blockDim.x) hs[k] = __ldcg(hsum + k);
  }
  __syncthreads();
  return true;
}

// ||h||^2 over hs[0 .. ncols), the same bits in every CTA: warp 0, then broadcast.
__device__ __forceinline__ double gm_hnorm2(const double* hs, int ncols, double* red) {
  if (threadIdx.x < 32) {
    double q = 0.0;
    for (int c = threadIdx.x; c < ncols; c += 32) q = fma(hs[c], hs[c], q);
    q = warp_sum(q);
    if (threadIdx.x == 0) red[0] = q;
  }
  __syncthreads();
  const double q = red[0];
  __syncthreads();
  return q;
}

// w[i] - sum_{c0 <= c < c1} V[c][i] h[c] for row i.  One chain: a warp issues one FP64 operation
// in 67 cycles whether or not the next depends on it, so interleaved chains only add the
// additions that join them.
__device__ __forceinline__ double gm_row_update(const double* __restrict__ V, int64_t ld, double wi,
                                                int64_t i, int c0, int c1, const double* hs) {
  int c = c0;
  for (; c + 7 < c1; c += 8) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = V[(int64_t)(c + k) * ld + i];
#pragma unroll
    for (int k = 0; k < 8; ++k) wi = fma(-v[k], hs[c + k], wi);
  }
  for (; c < c1; ++c) wi = fma(-V[(int64_t)c * ld + i], hs[c], wi);
  return wi;
}
__device__ __forceinline__ double gm_row_update(const double* __restrict__ V, int64_t ld, double wi,
                                                int64_t i, int ncols, const double* hs) {
  return gm_row_update(V, ld, wi, i, 0, ncols, hs);
}

// The same for rows i and i2 at once (same summation order as gm_row_update): 16 loads
// in flight per thread.
__device__ __forceinline__ void gm_row_update2(const double* __restrict__ V, int64_t ld, int64_t i,
                                               int64_t i2, int ncols, const double* hs, double& wa,
                                               double& wb) {
  int c = 0;
  for (; c + 7 < ncols; c += 8) {
    double va[8], vb[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      va[k] = V[(int64_t)(c + k) * ld + i];
      vb[k] = V[(int64_t)(c + k) * ld + i2];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      wa = fma(-va[k], hs[c + k], wa);
      wb = fma(-vb[k], hs[c + k], wb);
    }
  }
  for (; c < ncols; ++c) {
    wa = fma(-V[(int64_t)c * ld + i], hs[c], wa);
    wb = fma(-V[(int64_t)c * ld + i2], hs[c], wb);
  }
}

// SUMS = 1: the partials of the cluster's CTAs, part[c] in each one's shared memory, added in
// rank order by every CTA.
__device__ __forceinline__ void gm_cluster_sums(double* part, int cols, double* hs) {
  cl_sync();   // every CTA's partials are written
  for (int c = threadIdx.x; c < cols; c += blockDim.x) {
    double v[kGmCluster];
    const uint32_t a = smem_u32(part + c);
#pragma unroll
    for (int q = 0; q < kGmCluster; ++q)
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[q]) : "r"(cl_map(a, (uint32_t)q)) : "memory");
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < kGmCluster; ++q) s += v[q];
    hs[c] = s;
  }
  __syncthreads();
}

template <typename TAZ, bool WS, int SUMS>
__global__ void __launch_bounds__(kGmThreads, WS ? 1 : 2) gm_step_kernel(const GmStepArgs<TAZ> a) {
  if (a.st->done) return;   // uniform: read before any sync between CTAs
  extern __shared__ double wsm[];   // WS: w[r0 .. r1), then the staged columns
  __shared__ double hs[130];
  __shared__ double red[WS ? kGmRedWs : kGmRed];
  __shared__ double hcol[130];   // last CTA: the column j of the Hessenberg matrix
  __shared__ double pre[260];    // last CTA: what the Givens step reads
  __shared__ double part[SUMS == 1 ? 260 : 1];
  const int j = a.st->j, ncols = j + 1;
  // the last CTA has no rows: it does the Givens step, a chain of FP64 operations that would
  // wait behind its other warps' on the pipe
  const int nb = gridDim.x - 1, b = blockIdx.x;
  const bool giv = b == nb;
  const int64_t chunk = (a.len + nb - 1) / nb;
  const int64_t r0 = min(a.len, (int64_t)b * chunk), r1 = giv ? r0 : min(a.len, r0 + chunk);
  double* w = WS ? wsm - r0 : a.w;   // indexed by the row
  const double* V = a.V;
  int nfit = 0;
  const double* Vs = nullptr;        // staged columns, indexed by the row
  if constexpr (WS) {
    nfit = min(ncols, a.slab);
    if (nfit < ncols) nfit &= ~(kGmGroup - 1);
    double* slab = wsm + chunk;
    const int64_t vld = chunk | 1;
    const int rows = (int)(r1 - r0);
    for (int c = threadIdx.x >> 5; c < nfit; c += kGmThreads / 32)   // a warp per column
      for (int r = threadIdx.x & 31; r < rows; r += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(slab + (int64_t)c * vld + r)),
                     "l"(V + (int64_t)c * a.ld + r0 + r)
                     : "memory");
    Vs = slab - r0;
  }
  if (giv) gm_finish_prefetch(a.st, a.cs, a.sn, a.g, pre);
  {   // w_top = alpha v_top + A z (az; else w_top is formed in a.w), w_bot from a.w
    const double* vj = V + (int64_t)j * a.ld;
    const double al = a.alpha;
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
      if (a.az && i < a.m) w[i] = fma(al, vj[i], (double)a.az[i]);
      else if (WS) w[i] = a.w[i];
    }
    if constexpr (WS) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  // w1 = w - V h of row i
  auto project = [&](int64_t i, double wi) {
    if (nfit > 0) wi = gm_row_update(Vs, chunk | 1, wi, i, 0, nfit, hs);
    if (nfit < ncols) wi = gm_row_update(V, a.ld, wi, i, nfit, ncols, hs);
    return wi;
  };
  auto sums = [&](int which) -> bool {   // partials of V^T w and ||w||^2, added over the CTAs into hs
    if constexpr (SUMS == 1) {
      gm_partials(V, a.ld, Vs, chunk | 1, nfit, w, r0, r1, ncols, part + which * 130, 1, red, 0);
      gm_cluster_sums(part + which * 130, ncols + 1, hs);
      return true;
    } else {
      double* Dp = a.Dp + which * (a.ldd / 2);   // one half of every column of partials each
      gm_partials(V, a.ld, Vs, chunk | 1, nfit, w, r0, r1, ncols, Dp, a.ldd, red, blockIdx.x);
      return gm_grid_sums(Dp, a.ldd, a.hsum + which * (a.maxc + 1), ncols + 1, a.seq, which ? 0 : a.expire, a.err,
                          a.wait_ns, hs);
    }
  };
  // ---- first pass: h and ||w||^2
  if (!sums(0)) {
    if (threadIdx.x == 0) a.st->done = 1;   // later launches of the batch skip; the host reads err
    return;
  }
  const double wn2 = hs[ncols];
  const double hh = gm_hnorm2(hs, ncols, red);
  const bool second = hh > 0.5 * wn2;
  const int64_t step = blockDim.x;
  if (giv) {
    for (int c = threadIdx.x; c < ncols; c += blockDim.x) hcol[c] = hs[c];
    if (threadIdx.x == 0) {
      a.st->reorth = second ? 1 : 0;
      a.st->nreorth += second ? 1 : 0;
    }
  }
  double hn2;
  if (!second) {
    hn2 = wn2 - hh;
  } else {
    if constexpr (WS) {
      for (int64_t i = r0 + threadIdx.x; i < r1; i += step) w[i] = project(i, w[i]);
    } else {
      int64_t i = r0 + threadIdx.x;
      for (; i + step < r1; i += 2 * step) {
        double wa = w[i], wb = w[i + step];
        gm_row_update2(V, a.ld, i, i + step, ncols, hs, wa, wb);
        w[i] = wa;
        w[i + step] = wb;
      }
      for (; i < r1; i += step) w[i] = gm_row_update(V, a.ld, w[i], i, ncols, hs);
    }
    __syncthreads();   // this CTA's rows of w1 are final for the second pass
    if (!sums(1)) {
      if (threadIdx.x == 0) a.st->done = 1;   // later launches of the batch skip; the host reads err
      return;
    }
    if (giv)
      for (int c = threadIdx.x; c < ncols; c += blockDim.x) hcol[c] += hs[c];
    hn2 = hs[ncols] - gm_hnorm2(hs, ncols, red);
  }
  if (!(hn2 > 0.0)) hn2 = 0.0;
  // ---- the Givens step (last CTA) and the new column (own rows)
  if (giv) {
    __syncthreads();   // hcol is complete
    if (threadIdx.x < 32) gm_finish_warp(hn2, j, pre, a.st, hcol, a.H, a.ldh, a.cs, a.sn, a.g);
  } else {
    if (threadIdx.x < 32) {   // one warp: an FP64 reciprocal root
      const double v = hn2 > 0.0 ? rsqrt(hn2) : 0.0;
      if (threadIdx.x == 0) red[1] = v;
    }
    __syncthreads();
    const double inv = red[1];
    double* vn = a.V + (int64_t)(j + 1) * a.ld;
    int64_t i = r0 + threadIdx.x;
    if constexpr (!WS) {
      for (; i + step < r1; i += 2 * step) {
        double wa = w[i], wb = w[i + step];
        gm_row_update2(V, a.ld, i, i + step, ncols, hs, wa, wb);
        wa *= inv;
        wb *= inv;
        vn[i] = wa;
        vn[i + step] = wb;
        if (a.v32) {
          if (i < a.m) a.v32[i] = (float)wa;
          if (i + step < a.m) a.v32[i + step] = (float)wb;
        }
      }
    }
    for (; i < r1; i += step) {
      const double v = (WS ? project(i, w[i]) : gm_row_update(V, a.ld, w[i], i, ncols, hs)) * inv;
      vn[i] = v;
      if (a.v32 && i < a.m) a.v32[i] = (float)v;
    }
  }
  if constexpr (SUMS == 1) cl_sync();   // no CTA leaves while another may read its partials
}

// ---------------------------------------------------------------- MGS Arnoldi step
// Modified Gram-Schmidt in blocks of eight columns for long vectors, one cooperative launch
// per FGMRES iteration.  Sweep k = 0 .. K over the CTA's rows (K blocks): subtract the
// projection on block k-1 (its coefficients are the previous sweep's grid sums) and accumulate
// the eight products of block k with w (sweep K: ||w||^2); each sweep ends in one grid sum.
// 2(j+1) FP64 FMAs per row, the least any Gram-Schmidt form needs for j+1 projections
// (classical Gram-Schmidt with its second pass takes 4(j+1)); GB300's FP64 rate, not HBM,
// bounds the step at m in the millions.  Projecting on eight columns at once can leave
// the basis less orthogonal than one after the other does (||V^T V - I|| 0.9 to 2.3 times as large,
// emulated on the preconditioned augmented system, kappa 10 to 1e7); FGMRES takes the same iterations
// to the same residual.  It needs an eighth of the grid sums (about 4 us each: column by column,
// m = 1e6, j = 20 took 222 us a step, 152 us now, 67 us of them FMAs).
// Each row stays with one thread from sweep to sweep, so w needs no barrier between
// sweeps.  WS: the CTA's rows of w live in shared memory for the whole step (one CTA per
// SM; rows of [r; x] up to 152 x ~27,000), so a sweep reads only block k from HBM and block k-1
// again (from L2 while it fits); otherwise w is read and written in global memory every sweep.
constexpr int kMgsThreads = 512;
constexpr int kMgsStaticSmem = 16384; // bound on the kernels' static shared memory

// The grid sums of eight values: each CTA's part[c * ldd + block] (one fresh set of columns per
// sweep, so a CTA that has moved on disturbs no one still reading), added by a warp per column
// in block order in every CTA.  False if the wait ran out.
__device__ __forceinline__ bool gm_grid_sum8(const double* part, int ldd, int cols, unsigned long long* ctr,
                                             int plus_one, int* err, uint64_t wait_ns, double* out) {
  if (!gm_rendezvous(ctr, plus_one, err, wait_ns)) return false;
  const int nb = (int)gridDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < cols) {
    const double* col = part + (int64_t)warp * ldd;
    double t0 = 0.0, t1 = 0.0;
    int q = lane;
    for (; q + 32 < nb; q += 64) {
      t0 += __ldcg(col + q);
      t1 += __ldcg(col + q + 32);
    }
    if (q < nb) t0 += __ldcg(col + q);
    const double t = warp_sum(t0 + t1);
    if (lane == 0) out[warp] = t;
  }
  __syncthreads();
  return true;
}

template <typename TAZ, bool WS>
__global__ void __launch_bounds__(kMgsThreads, WS ? 1 : 2) gm_mgs_kernel(const GmStepArgs<TAZ> a) {
  if (a.st->done) return;   // uniform: read before any grid sync
  extern __shared__ double wsm[];   // WS: w[r0 .. r1)
  __shared__ double hs[144];        // the coefficients; zero past ncols up to a whole block
  __shared__ double red[kMgsThreads / 32][kGmGroup + 1];
  __shared__ double hcol[130];
  __shared__ double pre[260];
  __shared__ double wn2_s, inv_s;
  const int j = a.st->j, ncols = j + 1;
  const int K = (ncols + kGmGroup - 1) / kGmGroup;
  const int nb = gridDim.x - 1, b = blockIdx.x;   // the last CTA: the Givens step, no rows
  const bool giv = b == nb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t chunk = (a.len + nb - 1) / nb;
  const int64_t r0 = min(a.len, (int64_t)b * chunk), r1 = giv ? r0 : min(a.len, r0 + chunk);
  constexpr int64_t step = kMgsThreads;
  double* w = WS ? wsm - r0 : a.w;   // indexed by the row
  const double* wg = a.w;
  const double* V = a.V;
  const double* vj = V + (int64_t)j * a.ld;
  const double al = a.alpha;
  const bool form = a.az != nullptr;
  if (giv) gm_finish_prefetch(a.st, a.cs, a.sn, a.g, pre);
  for (int k = 0; k <= K; ++k) {
    // block k - 1 subtracted, block k accumulated; columns past ncols are read as column 0 with a
    // zero coefficient, and their sums dropped
    const double* vp[kGmGroup];
    const double* vc[kGmGroup];
    double hp[kGmGroup], t[kGmGroup];
#pragma unroll
    for (int q = 0; q < kGmGroup; ++q) {
      const int cp = (k - 1) * kGmGroup + q, cc = k * kGmGroup + q;
      vp[q] = V + (k > 0 && cp < ncols ? (int64_t)cp * a.ld : 0);
      vc[q] = V + (cc < ncols ? (int64_t)cc * a.ld : 0);
      hp[q] = (k > 0 && cp < ncols) ? -hs[cp] : 0.0;
      t[q] = 0.0;
    }
    const int np = k > 0 ? min(kGmGroup, ncols - (k - 1) * kGmGroup) : 0;
    const int nc = k < K ? min(kGmGroup, ncols - k * kGmGroup) : 0;
    for (int64_t i = r0 + threadIdx.x; i < r1; i += step) {
      double pv[kGmGroup], cv[kGmGroup];
      double wi = k > 0 ? w[i] : ((form && i < a.m) ? fma(al, vj[i], (double)a.az[i]) : wg[i]);
#pragma unroll
      for (int q = 0; q < kGmGroup; ++q) pv[q] = q < np ? vp[q][i] : 0.0;
#pragma unroll
      for (int q = 0; q < kGmGroup; ++q) cv[q] = q < nc ? vc[q][i] : 0.0;
      if (k > 0) {
        double p0 = 0.0, p1 = 0.0;
#pragma unroll
        for (int q = 0; q < kGmGroup; q += 2) {
          if (q < np) p0 = fma(hp[q], pv[q], p0);
          if (q + 1 < np) p1 = fma(hp[q + 1], pv[q + 1], p1);
        }
        wi += p0 + p1;
      }
      if (WS || k > 0 || (form && i < a.m)) w[i] = wi;
      if (k < K) {
#pragma unroll
        for (int q = 0; q < kGmGroup; ++q)
          if (q < nc) t[q] = fma(cv[q], wi, t[q]);
      } else {
        t[0] = fma(wi, wi, t[0]);
      }
    }
    const double tot = warp_reduce8(t);
    __syncthreads();   // the previous sweep's red has been read
    if ((lane & 3) == 0) red[warp][(lane >> 2) & 7] = tot;
    __syncthreads();
    const int cols = k < K ? nc : 1;
    double* part = a.Dp + (int64_t)k * kGmGroup * a.ldd;
    if (threadIdx.x < cols) {
      double s0 = 0.0, s1 = 0.0;
#pragma unroll
      for (int q = 0; q < kMgsThreads / 32; q += 2) {
        s0 += red[q][threadIdx.x];
        s1 += red[q + 1][threadIdx.x];
      }
      part[(int64_t)threadIdx.x * a.ldd + b] = s0 + s1;
    }
    if (!gm_grid_sum8(part, a.ldd, cols, a.seq, a.expire, a.err, a.wait_ns, k < K ? hs + k * kGmGroup : &wn2_s)) {
      if (threadIdx.x == 0) a.st->done = 1;   // later launches of the batch skip; the host reads err
      return;
    }
  }
  double hn2 = wn2_s;
  if (!(hn2 > 0.0)) hn2 = 0.0;
  if (giv) {
    for (int c = threadIdx.x; c < ncols; c += blockDim.x) hcol[c] = hs[c];
    if (threadIdx.x == 0) a.st->reorth = 0;
    __syncthreads();
    if (threadIdx.x < 32) gm_finish_warp(hn2, j, pre, a.st, hcol, a.H, a.ldh, a.cs, a.sn, a.g);
    return;
  }
  if (threadIdx.x < 32) {   // one warp: an FP64 reciprocal root
    const double v = hn2 > 0.0 ? rsqrt(hn2) : 0.0;
    if (threadIdx.x == 0) inv_s = v;
  }
  double* vn = a.V + (int64_t)(j + 1) * a.ld;
  __syncthreads();   // every thread's last w is visible to the CTA
  const double inv = inv_s;
  for (int64_t i = r0 + threadIdx.x; i < r1; i += step) {
    const double v = w[i] * inv;
    vn[i] = v;
    if (a.v32 && i < a.m) a.v32[i] = (float)v;
  }
}

// Shared memory for w and the staged columns.
constexpr size_t kGmRoom = 227 * 1024 - kMgsStaticSmem;

// Clusters of kGmCluster CTAs that fit the device with all of kGmRoom (a non-portable size: none where
// sixteen SMs of one group are not to be had, as in a slice of the GPU).
template <typename TAZ>
static int gm_clusters() {
  auto kern = gm_step_kernel<TAZ, true, 1>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kGmCluster);
  cfg.blockDim = dim3(kGmThreads);
  cfg.dynamicSmemBytes = kGmRoom;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kGmCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (allow_dyn_smem(kern, kGmRoom) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();   // no such clusters: the grid form serves
    return 0;
  }
  return clusters;
}

template <typename TAZ>
cudaError_t launch_gm_step(double* V, int64_t ld, double* w, int64_t len, int64_t m, const TAZ* az,
                           GmState* st, int maxc, double* Dp, double* hsum, double* H, int ldh,
                           double* cs, double* sn, double* g, float* v32, int* err,
                           int num_sms, cudaStream_t s, uint64_t wait_ns, double alpha, int gs,
                           unsigned long long* seq, int expire) {
  static_assert(sizeof(GmStepArgs<TAZ>) < 4096, "kernel parameter block");
  if (maxc > 128 || gs < 0 || gs > 2 || seq == nullptr) return cudaErrorInvalidValue;
  const bool mgs = gs > 0;
  // Classical: up to kGmClusterRows rows one cluster of sixteen CTAs (gm_one_cluster); up to 2^20 a
  // cooperative launch of at most one CTA per 64 rows and SM; both with w and the basis columns that fit in
  // shared memory.  From 2^20 rows on (opts.arnoldi = 1) two CTAs per SM with w in global memory
  // (more loads in flight).  Modified: one per SM with w in shared memory where one CTA's rows
  // fit (unless gs = 2), else as classical; the last CTA of every form has no rows.
  const bool lng = len >= ((int64_t)1 << 20);
  const bool cl = gm_one_cluster(len, gs, expire, 1) && gm_one_cluster(len, gs, expire, gm_clusters<TAZ>());
  const int64_t cgs_blk = cl ? kGmCluster : std::max<int64_t>(2, std::min<int64_t>(num_sms, (len + 63) / 64 + 1));
  const int64_t row_ctas = mgs ? std::max(1, num_sms - 1) : cgs_blk - 1;
  const int64_t ws_rows = (len + row_ctas - 1) / row_ctas;
  const size_t ws_bytes = (size_t)ws_rows * 8;
  const bool ws = mgs ? (gs == 1 && ws_bytes <= kGmRoom) : !lng;
  auto kern = !mgs ? (cl ? gm_step_kernel<TAZ, true, 1> : (ws ? gm_step_kernel<TAZ, true, 0> : gm_step_kernel<TAZ, false, 0>))
                   : (ws ? gm_mgs_kernel<TAZ, true> : gm_mgs_kernel<TAZ, false>);
  const int threads = mgs ? kMgsThreads : kGmThreads;
  // staged columns (classical): all maxc, or as many as fit beside w
  const size_t col_bytes = (size_t)(ws_rows | 1) * 8;
  const int slab = (!mgs && ws && ws_bytes < kGmRoom) ? (int)std::min<int64_t>(maxc, (int64_t)((kGmRoom - ws_bytes) / col_bytes)) : 0;
  const size_t dyn = ws ? ws_bytes + col_bytes * (size_t)slab : 0;
  if (ws) {
    cudaError_t e = allow_dyn_smem(kern, dyn);
    if (e != cudaSuccess) return e;
  }
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, dyn);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  const int nblk = ws ? (int)row_ctas + 1 : std::max(2, num_sms * (occ >= 2 && lng ? 2 : 1));
  GmStepArgs<TAZ> a{V, ld, len, m, w, az, st, maxc, 0, Dp, hsum, H, cs, sn, g, v32, err};
  a.ldh = ldh;
  a.ldd = 4 * num_sms;   // the caller's Dp holds (maxc + 17) x 4 num_sms values
  a.wait_ns = wait_ns > 0 ? wait_ns : kWaitLimitNs;
  a.alpha = alpha;
  a.seq = seq;
  a.expire = expire;
  a.slab = slab;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nblk);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (cl) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kGmCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}
template cudaError_t launch_gm_step<float>(double*, int64_t, double*, int64_t, int64_t, const float*, GmState*,
                                           int, double*, double*, double*, int, double*, double*,
                                           double*, float*, int*, int, cudaStream_t, uint64_t, double, int,
                                           unsigned long long*, int);
template cudaError_t launch_gm_step<double>(double*, int64_t, double*, int64_t, int64_t, const double*,
                                            GmState*, int, double*, double*, double*, int, double*,
                                            double*, double*, float*, int*, int, cudaStream_t, uint64_t, double,
                                            int, unsigned long long*, int);

// y = H[:k,:k]^-1 g[:k] (k <= 128): column-oriented back substitution by one warp, the right-hand
// side in registers.  H comes in by 128 threads and the diagonal's reciprocals are formed side
// by side, since an FP64 quotient is a chain of some 500 cycles: yi = a / d is a product and one
// residual correction (a / d itself where 1 / d is not finite or zero).  With the quotients in
// the chain and one warp's loads k = 40 took 57 us, 25 now.
constexpr int kGmSolveThreads = 128;
__device__ __forceinline__ void gm_solve_body(int k, const double* __restrict__ H, int ldh,
                                              const double* __restrict__ g, double* __restrict__ y, double* hs) {
  __shared__ double rinv[kGmSolveThreads];
  const int tid = threadIdx.x;
#pragma unroll 4
  for (int e = tid; e < k * k; e += kGmSolveThreads) {
    const int c = e / k, i = e % k;
    hs[e] = i <= c ? H[(int64_t)c * ldh + i] : 0.0;
  }
  if (tid < k) rinv[tid] = 1.0 / H[(int64_t)tid * ldh + tid];
  __syncthreads();
  if (tid >= 32) return;
  constexpr int NQ = kGmSolveThreads / 32;
  double x[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) x[q] = tid + 32 * q < k ? g[tid + 32 * q] : 0.0;
#pragma unroll
  for (int q = NQ - 1; q >= 0; --q) {
    for (int ii = min(31, k - 1 - 32 * q); ii >= 0; --ii) {
      const int i = 32 * q + ii;
      const double* col = hs + (size_t)i * k;
      const double a = __shfl_sync(0xffffffffu, x[q], ii), d = col[i], ri = rinv[i];
      double yi = a * ri;
      yi = fma(fma(-yi, d, a), ri, yi);
      if (!(fabs(ri) > 0.0 && fabs(ri) <= 1.7976931348623157e308)) yi = a / d;
#pragma unroll
      for (int p = 0; p <= q; ++p)
        if (tid + 32 * p < i) x[p] = fma(-col[tid + 32 * p], yi, x[p]);
      if (tid == 0) y[i] = yi;
    }
  }
}
__global__ void __launch_bounds__(kGmSolveThreads)
    gm_solve_kernel(const GmState* st, const double* H, int ldh, const double* g, double* y) {
  extern __shared__ double hs[];   // k x k, column-major
  gm_solve_body(st->j, H, ldh, g, y, hs);
}

// d[i] += sum_c B[c][i] y[c] for i < len (B column-major, ld); partial sums of
// the correction squared and of the updated vector squared.
template <typename TB>
__global__ void gm_apply_kernel(const TB* __restrict__ B, int64_t ld, int64_t len, const GmState* st,
                                const double* __restrict__ y, double* __restrict__ d,
                                double* part_dd, double* part_d, double scale) {
  __shared__ double ys[128];
  __shared__ double red[33];
  const int k = st->j;
  for (int c = threadIdx.x; c < k; c += blockDim.x) ys[c] = y[c];
  __syncthreads();
  double s1 = 0.0, s2 = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x) {
    // four interleaved chains, their loads issued together (the loop is latency-bound)
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    int c = 0;
    for (; c + 3 < k; c += 4) {
      const TB* bc = B + (int64_t)c * ld + i;
      const double b0 = (double)bc[0], b1 = (double)bc[ld], b2 = (double)bc[2 * ld], b3 = (double)bc[3 * ld];
      a0 = fma(b0, ys[c], a0);
      a1 = fma(b1, ys[c + 1], a1);
      a2 = fma(b2, ys[c + 2], a2);
      a3 = fma(b3, ys[c + 3], a3);
    }
    for (; c < k; ++c) a0 = fma((double)B[(int64_t)c * ld + i], ys[c], a0);
    double acc = ((a0 + a1) + (a2 + a3)) * scale;
    const double nv = d[i] + acc;
    d[i] = nv;
    s1 += acc * acc;
    s2 += nv * nv;
  }
  s1 = block_sum_d(s1, red);
  s2 = block_sum_d(s2, red);
  if (threadIdx.x == 0) {
    part_dd[blockIdx.x] = s1;
    part_d[blockIdx.x] = s2;
  }
}

cudaError_t launch_gm_init(const double* sq_partial, int nblk, GmState* st, double* g, cudaStream_t s) {
  gm_init_kernel<<<1, 256, 0, s>>>(sq_partial, nblk, st, g);
  return cudaGetLastError();
}
cudaError_t launch_gm_solve(const GmState* st, const double* H, int ldh, const double* g, double* y,
                            cudaStream_t s) {
  const size_t smem = (size_t)(ldh - 1) * (ldh - 1) * sizeof(double);
  if (smem > 48 * 1024) {
    cudaError_t e = allow_dyn_smem(gm_solve_kernel, smem);
    if (e != cudaSuccess) return e;
  }
  gm_solve_kernel<<<1, kGmSolveThreads, smem, s>>>(st, H, ldh, g, y);
  return cudaGetLastError();
}
template <typename TB>
cudaError_t launch_gm_apply(const TB* B, int64_t ld, int64_t len, const GmState* st, const double* y,
                            double* d, double* part_dd, double* part_d, int nblk, cudaStream_t s,
                            double scale) {
  gm_apply_kernel<TB><<<nblk, 256, 0, s>>>(B, ld, len, st, y, d, part_dd, part_d, scale);
  return cudaGetLastError();
}
template cudaError_t launch_gm_apply<double>(const double*, int64_t, int64_t, const GmState*, const double*,
                                             double*, double*, double*, int, cudaStream_t, double);
template cudaError_t launch_gm_apply<float>(const float*, int64_t, int64_t, const GmState*, const double*,
                                            double*, double*, double*, int, cudaStream_t, double);

cudaError_t launch_sum_partials(const double* partial, int nblk, double* out, bool take_sqrt,
                                cudaStream_t st) {
  sum_partials_kernel<<<1, 1024, 0, st>>>(partial, nblk, out, take_sqrt);
  return cudaGetLastError();
}

// Copies [f; h] into V[:, 0] and leaves partial sums of squares.
__global__ void gm_rhs_kernel(const double* __restrict__ f, const double* __restrict__ h, int64_t m,
                              int64_t n, double* __restrict__ V0, double* sq_partial, double alpha) {
  __shared__ double red[33];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m + n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = (i < m) ? f[i] : (alpha == 1.0 ? h[i - m] : h[i - m] / alpha);
    V0[i] = v;
    s += v * v;
  }
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) sq_partial[blockIdx.x] = s;
}

cudaError_t launch_gm_rhs(const double* f, const double* h, int64_t m, int64_t n, double* V0,
                          double* sq_partial, int nblk, cudaStream_t s, double alpha) {
  gm_rhs_kernel<<<nblk, 256, 0, s>>>(f, h, m, n, V0, sq_partial, alpha);
  return cudaGetLastError();
}

// V[:, 0] *= inv_h (after gm_init)
__global__ void gm_scale0_kernel(double* V0, int64_t len, const GmState* st, float* v32, int64_t m) {
  const double s = st->inv_h;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = V0[i] * s;
    V0[i] = v;
    if (v32 && i < m) v32[i] = (float)v;
  }
}
cudaError_t launch_gm_scale0(double* V0, int64_t len, const GmState* st, float* v32, int64_t m,
                             int nblk, cudaStream_t s) {
  gm_scale0_kernel<<<nblk, 256, 0, s>>>(V0, len, st, v32, m);
  return cudaGetLastError();
}


// ============================================================ grouped (batched) forms
// Problem p owns CTAs [start[p], start[p + 1]) of each launch; its block index and
// block count within the launch stand in for blockIdx.x and gridDim.x of the
// single-problem kernels above, whose bodies these call.

// Persistent over the items (problem, block of the problem's pass): CTA b takes items b,
// b + gridDim.x, ...; every item is computed exactly as a CTA of that problem's own pass
// would compute it, so the result does not depend on the grid size.
template <typename T, int VW, int VPL, int MODE>
__global__ void __launch_bounds__(256)
    grouped_pass_kernel(const PassArgs<T>* __restrict__ tab, const int* __restrict__ start, int nprob,
                        int64_t items) {
  for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const int pr = group_of(start, nprob, it);
    pass_ring_body<T, VW, VPL, MODE>(tab[pr], it - start[pr], (int64_t)start[pr + 1] - start[pr]);
    __syncthreads();   // the item's shared-memory reduction is read before the next item writes it
  }
}

template <typename T>
cudaError_t launch_grouped_pass(int mode, int vw, int vpl, const PassArgs<T>* tab, const int* start,
                                int64_t ctas, int nprob, size_t smem, cudaStream_t st, int64_t grid) {
  if (ctas <= 0) return cudaSuccess;
  if (ctas > 2147483647LL) return cudaErrorInvalidValue;
  const int64_t g = (grid > 0 && grid < ctas) ? grid : ctas;
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_dyn_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)g, 256, smem, st>>>(tab, start, nprob, ctas);
    return cudaGetLastError();
  };
  smem *= 2 * kRingPairs;   // the caller's size is 8 warps x one row
  if constexpr (sizeof(T) == 4) {
    if (vw != 4 || vpl != 2) return cudaErrorInvalidValue;
    if (mode == PM_LSQR) return go(grouped_pass_kernel<float, 4, 2, PM_LSQR>);
    if (mode == PM_FGM) return go(grouped_pass_kernel<float, 4, 2, PM_FGM>);
  } else {
    if (vw != 1 || vpl != 8) return cudaErrorInvalidValue;
    if (mode == PM_LSQR) return go(grouped_pass_kernel<double, 1, 8, PM_LSQR>);
    if (mode == PM_FGM) return go(grouped_pass_kernel<double, 1, 8, PM_FGM>);
    if (mode == PM_RES) return go(grouped_pass_kernel<double, 1, 8, PM_RES>);
  }
  return cudaErrorInvalidValue;
}
template cudaError_t launch_grouped_pass<float>(int, int, int, const PassArgs<float>*, const int*, int64_t, int,
                                                size_t, cudaStream_t, int64_t);
template cudaError_t launch_grouped_pass<double>(int, int, int, const PassArgs<double>*, const int*, int64_t, int,
                                                 size_t, cudaStream_t, int64_t);

template <typename TP, typename TO>
__global__ void grouped_colsum_kernel(const GColsum<TP, TO>* __restrict__ tab, const int* __restrict__ start,
                                      int nprob) {
  const int pr = group_of(start, nprob, blockIdx.x);
  const GColsum<TP, TO>& g = tab[pr];
  colsum_body<TP, TO>(g.P, g.nblk, g.n, g.scale_ptr, g.scale_mul, g.out, g.done, (int64_t)blockIdx.x - start[pr]);
}

template <typename TP, typename TO>
cudaError_t launch_grouped_colsum(const GColsum<TP, TO>* tab, const int* start, int64_t ctas, int nprob,
                                  cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  grouped_colsum_kernel<TP, TO><<<(unsigned)ctas, kColsumCols * 32, 0, st>>>(tab, start, nprob);
  return cudaGetLastError();
}
template cudaError_t launch_grouped_colsum<float, float>(const GColsum<float, float>*, const int*, int64_t, int,
                                                         cudaStream_t);
template cudaError_t launch_grouped_colsum<double, double>(const GColsum<double, double>*, const int*, int64_t,
                                                           int, cudaStream_t);

template <typename TP>
__global__ void grouped_lsqr_colsum_kernel(const GLsqrColsum<TP>* __restrict__ tab, const int* __restrict__ start,
                                           int nprob, bool init) {
  const int pr = group_of(start, nprob, blockIdx.x);
  const GLsqrColsum<TP>& g = tab[pr];
  lsqr_colsum_body<TP>(g.P, g.nblk, g.n, g.sq, g.st, init, g.out, (int64_t)blockIdx.x - start[pr]);
}

template <typename TP>
cudaError_t launch_grouped_lsqr_colsum(const GLsqrColsum<TP>* tab, const int* start, int64_t ctas, int nprob,
                                       bool init, cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  grouped_lsqr_colsum_kernel<TP><<<(unsigned)ctas, (kColsumCols + 1) * 32, 0, st>>>(tab, start, nprob, init);
  return cudaGetLastError();
}
template cudaError_t launch_grouped_lsqr_colsum<float>(const GLsqrColsum<float>*, const int*, int64_t, int, bool,
                                                       cudaStream_t);

template <typename T>
__global__ void __launch_bounds__(kTrsvThreads)
    grouped_lsqr_step_kernel(const GLsqrStep<T>* __restrict__ tab, bool init) {
  const GLsqrStep<T>& g = tab[blockIdx.x];
  lsqr_step_body<T>(g.f, g.s, g.v, g.w, g.z, g.t, g.st, init);
}

template <typename T>
cudaError_t launch_grouped_lsqr_step(const GLsqrStep<T>* tab, int nprob, bool init, cudaStream_t st) {
  if (nprob <= 0) return cudaSuccess;
  const size_t smem = TrsvSmem<T>::bytes;
  cudaError_t e = allow_dyn_smem(grouped_lsqr_step_kernel<T>, smem);
  if (e != cudaSuccess) return e;
  grouped_lsqr_step_kernel<T><<<(unsigned)nprob, kTrsvThreads, smem, st>>>(tab, init);
  return cudaGetLastError();
}
template cudaError_t launch_grouped_lsqr_step<float>(const GLsqrStep<float>*, int, bool, cudaStream_t);

template <typename TX, typename TY, typename TO>
__global__ void grouped_axpby_kernel(const GAxpby<TX, TY, TO>* __restrict__ tab, const int* __restrict__ start,
                                     int nprob) {
  const int pr = group_of(start, nprob, blockIdx.x);
  const GAxpby<TX, TY, TO>& g = tab[pr];
  if (g.done && *g.done) return;
  const int64_t i = ((int64_t)blockIdx.x - start[pr]) * blockDim.x + threadIdx.x;
  if (i >= g.len) return;
  double v = (double)g.x[i] * g.a;
  if (g.y) v += (double)g.y[i] * g.b;
  g.out[i] = (TO)v;
}

template <typename TX, typename TY, typename TO>
cudaError_t launch_grouped_axpby(const GAxpby<TX, TY, TO>* tab, const int* start, int64_t ctas, int nprob,
                                 cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  grouped_axpby_kernel<TX, TY, TO><<<(unsigned)ctas, 256, 0, st>>>(tab, start, nprob);
  return cudaGetLastError();
}
template cudaError_t launch_grouped_axpby<double, double, float>(const GAxpby<double, double, float>*, const int*,
                                                                 int64_t, int, cudaStream_t);
template cudaError_t launch_grouped_axpby<float, double, double>(const GAxpby<float, double, double>*, const int*,
                                                                 int64_t, int, cudaStream_t);
template cudaError_t launch_grouped_axpby<double, double, double>(const GAxpby<double, double, double>*,
                                                                  const int*, int64_t, int, cudaStream_t);

// ||x|| by one CTA per problem
__global__ void grouped_norm_kernel(const GNorm* __restrict__ tab) {
  __shared__ double red[33];
  const GNorm& g = tab[blockIdx.x];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < g.len; i += blockDim.x) s += g.x[i] * g.x[i];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) *g.out = sqrt(s);
}

cudaError_t launch_grouped_norm(const GNorm* tab, int nprob, cudaStream_t st) {
  if (nprob <= 0) return cudaSuccess;
  grouped_norm_kernel<<<(unsigned)nprob, 1024, 0, st>>>(tab);
  return cudaGetLastError();
}

// ---- FGMRES
// rhs: V[:, 0] = [f; h / alpha] over the problem's CTAs, partial sums of squares
__global__ void grouped_gm_rhs_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob) {
  __shared__ double red[33];
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  double s = 0.0;
  if (!*g.skip) {
    for (int64_t i = blk * blockDim.x + threadIdx.x; i < g.m + g.n; i += nb * blockDim.x) {
      const double v = (i < g.m) ? g.f[i] : (g.alpha == 1.0 ? g.h[i - g.m] : g.h[i - g.m] / g.alpha);
      g.V[i] = v;
      s += v * v;
    }
  }
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) g.sqp[blk] = s;
}

// beta = ||[f; h / alpha]|| (partials in CTA order), state reset, g = beta e_1
__global__ void grouped_gm_init_kernel(const GGm* __restrict__ tab, const int* __restrict__ start) {
  __shared__ double red[33];
  const GGm& g = tab[blockIdx.x];
  const int nb = start[blockIdx.x + 1] - start[blockIdx.x];
  double s = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) s += g.sqp[b];
  s = block_sum_d(s, red);
  if (threadIdx.x == 0) {
    GmState* st = g.st;
    const double beta = sqrt(s);
    st->beta0 = beta;
    st->inv_h = beta > 0.0 ? 1.0 / beta : 0.0;
    st->j = 0;
    st->relres = beta > 0.0 ? 1.0 : 0.0;
    st->reorth = 0;
    st->nreorth = 0;
    st->done = (*g.skip || beta == 0.0 || st->maxit <= 0) ? 1 : 0;
    g.g[0] = beta;
  }
}

__global__ void grouped_gm_scale0_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob) {
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  if (g.st->done) return;
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  const double sc = g.st->inv_h;
  for (int64_t i = blk * blockDim.x + threadIdx.x; i < g.m + g.n; i += nb * blockDim.x) {
    const double v = g.V[i] * sc;
    g.V[i] = v;
    if (g.v32 && i < g.m) g.v32[i] = (float)v;
  }
}

cudaError_t launch_grouped_gm_init(const GGm* tab, const int* start, int64_t ctas, int nprob, cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  grouped_gm_rhs_kernel<<<(unsigned)ctas, 256, 0, st>>>(tab, start, nprob);
  grouped_gm_init_kernel<<<(unsigned)nprob, 256, 0, st>>>(tab, start);
  grouped_gm_scale0_kernel<<<(unsigned)ctas, 256, 0, st>>>(tab, start, nprob);
  return cudaGetLastError();
}

// Arnoldi, phase A (second = 0): w_top = alpha v_top + A z (unless the pass formed it), then
// the partials of V^T w and ||w||^2 over the CTA's rows; phase A' (second = 1, problems
// whose first pass lost more than half of ||w||^2): the same partials of w1.
__global__ void __launch_bounds__(kGmThreads)
    garn_partials_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob, int second) {
  __shared__ double red[kGmRed];
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  const GmState* st = g.st;
  if (st->done || (second && !st->reorth)) return;
  const int j = st->j, ncols = j + 1;
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  const int64_t len = g.m + g.n, chunk = (len + nb - 1) / nb;
  const int64_t r0 = blk * chunk, r1 = min(len, r0 + chunk);
  if (!second && g.az) {
    const double* vj = g.V + (int64_t)j * g.ld;
    const double al = g.alpha;
    for (int64_t i = r0 + threadIdx.x; i < min(r1, g.m); i += blockDim.x) {
      const double azi = g.az_f32 ? (double)static_cast<const float*>(g.az)[i] : static_cast<const double*>(g.az)[i];
      g.w[i] = fma(al, vj[i], azi);
    }
    __syncthreads();
  }
  gm_partials(g.V, g.ld, nullptr, 0, 0, g.w, r0, r1, ncols, g.Dp, (int)nb, red, blk);
}

// phase B / B' (one CTA per problem): column sums of the partials in block order, then the
// twice-is-enough test (first pass) and the squared norm of the new column
__global__ void __launch_bounds__(kGmThreads)
    garn_reduce_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int second) {
  const GGm& g = tab[blockIdx.x];
  GmState* st = g.st;
  if (st->done || (second && !st->reorth)) return;
  const int j = st->j, ncols = j + 1;
  const int nb = start[blockIdx.x + 1] - start[blockIdx.x];
  double* hs = second ? g.hs2 : g.hs1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int c = warp; c <= ncols; c += nw) {
    const double* col = g.Dp + (int64_t)c * nb;
    double t0 = 0.0, t1 = 0.0;
    int q = lane;
    for (; q + 32 < nb; q += 64) {
      t0 += col[q];
      t1 += col[q + 32];
    }
    if (q < nb) t0 += col[q];
    const double tt = warp_sum(t0 + t1);
    if (lane == 0) hs[c] = tt;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double q = 0.0;
    for (int c = 0; c < ncols; ++c) q = fma(hs[c], hs[c], q);
    const double wn2 = hs[ncols];
    if (!second) {
      const int re = q > 0.5 * wn2 ? 1 : 0;
      st->reorth = re;
      st->nreorth += re;
      const double hn2 = wn2 - q;
      g.hs1[ncols + 1] = hn2 > 0.0 ? hn2 : 0.0;   // used when there is no second pass
    } else {
      const double hn2 = wn2 - q;
      g.hs2[ncols + 1] = hn2 > 0.0 ? hn2 : 0.0;
    }
  }
}

// phase C1 (second pass problems): w1 = w - V h over the CTA's rows
__global__ void __launch_bounds__(kGmThreads)
    garn_sub_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob) {
  __shared__ double hs[130];
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  const GmState* st = g.st;
  if (st->done || !st->reorth) return;
  const int j = st->j, ncols = j + 1;
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  const int64_t len = g.m + g.n, chunk = (len + nb - 1) / nb;
  const int64_t r0 = blk * chunk, r1 = min(len, r0 + chunk);
  for (int c = threadIdx.x; c < ncols; c += blockDim.x) hs[c] = g.hs1[c];
  __syncthreads();
  const int64_t step = blockDim.x;
  int64_t i = r0 + threadIdx.x;
  for (; i + step < r1; i += 2 * step) {
    double wa = g.w[i], wb = g.w[i + step];
    gm_row_update2(g.V, g.ld, i, i + step, ncols, hs, wa, wb);
    g.w[i] = wa;
    g.w[i + step] = wb;
  }
  for (; i < r1; i += step) g.w[i] = gm_row_update(g.V, g.ld, g.w[i], i, ncols, hs);
}

// phase C: v_{j+1} = (w - V h) / ||w - V h|| over the CTA's rows (h of the last pass)
__global__ void __launch_bounds__(kGmThreads)
    garn_newcol_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob) {
  __shared__ double hs[130];
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  const GmState* st = g.st;
  if (st->done) return;
  const int j = st->j, ncols = j + 1;
  const double* hsrc = st->reorth ? g.hs2 : g.hs1;
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  const int64_t len = g.m + g.n, chunk = (len + nb - 1) / nb;
  const int64_t r0 = blk * chunk, r1 = min(len, r0 + chunk);
  for (int c = threadIdx.x; c < ncols; c += blockDim.x) hs[c] = hsrc[c];
  if (threadIdx.x < 32) {   // one warp: an FP64 root and quotient
    const double hn2 = hsrc[ncols + 1];
    const double v = hn2 > 0.0 ? rsqrt(hn2) : 0.0;
    if (threadIdx.x == 0) hs[ncols] = v;
  }
  __syncthreads();
  const double inv = hs[ncols];
  double* vn = g.V + (int64_t)(j + 1) * g.ld;
  const int64_t step = blockDim.x;
  int64_t i = r0 + threadIdx.x;
  for (; i + step < r1; i += 2 * step) {
    double wa = g.w[i], wb = g.w[i + step];
    gm_row_update2(g.V, g.ld, i, i + step, ncols, hs, wa, wb);
    wa *= inv;
    wb *= inv;
    vn[i] = wa;
    vn[i + step] = wb;
    if (g.v32) {
      if (i < g.m) g.v32[i] = (float)wa;
      if (i + step < g.m) g.v32[i + step] = (float)wb;
    }
  }
  for (; i < r1; i += step) {
    const double v = gm_row_update(g.V, g.ld, g.w[i], i, ncols, hs) * inv;
    vn[i] = v;
    if (g.v32 && i < g.m) g.v32[i] = (float)v;
  }
}

// phase D (one warp per problem): Hessenberg column h (+ h2), Givens step, j + 1
__global__ void garn_finish_kernel(const GGm* __restrict__ tab) {
  __shared__ double hcol[130];
  __shared__ double pre[260];
  const GGm& g = tab[blockIdx.x];
  GmState* st = g.st;
  if (st->done) return;
  const int j = st->j, ncols = j + 1;
  const int re = st->reorth;
  gm_finish_prefetch(st, g.cs, g.sn, g.g, pre);
  for (int c = threadIdx.x; c < ncols; c += 32) hcol[c] = re ? g.hs1[c] + g.hs2[c] : g.hs1[c];
  __syncwarp();
  const double hn2 = re ? g.hs2[ncols + 1] : g.hs1[ncols + 1];
  gm_finish_warp(hn2, j, pre, st, hcol, g.H, g.ldh, g.cs, g.sn, g.g);
}

cudaError_t launch_grouped_arnoldi(const GGm* tab, const int* start, int64_t ctas, int nprob, cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  const unsigned nc = (unsigned)ctas, np = (unsigned)nprob;
  garn_partials_kernel<<<nc, kGmThreads, 0, st>>>(tab, start, nprob, 0);
  garn_reduce_kernel<<<np, kGmThreads, 0, st>>>(tab, start, 0);
  garn_sub_kernel<<<nc, kGmThreads, 0, st>>>(tab, start, nprob);
  garn_partials_kernel<<<nc, kGmThreads, 0, st>>>(tab, start, nprob, 1);
  garn_reduce_kernel<<<np, kGmThreads, 0, st>>>(tab, start, 1);
  garn_newcol_kernel<<<nc, kGmThreads, 0, st>>>(tab, start, nprob);
  garn_finish_kernel<<<np, 32, 0, st>>>(tab);
  return cudaGetLastError();
}

// update: y = H^-1 g (one CTA per problem), then r += alpha V_top y, x += Z y over the
// problem's CTAs with the partial sums of ||alpha V_top y||^2, ||r||^2, ||Z y||^2, ||x||^2
__global__ void __launch_bounds__(kGmSolveThreads) grouped_gm_solve_kernel(const GGm* __restrict__ tab) {
  extern __shared__ double hsm[];   // k x k, column-major
  const GGm& g = tab[blockIdx.x];
  if (*g.skip) return;
  gm_solve_body(g.st->j, g.H, g.ldh, g.g, g.y, hsm);
}

__global__ void grouped_gm_apply_kernel(const GGm* __restrict__ tab, const int* __restrict__ start, int nprob) {
  __shared__ double ys[128];
  __shared__ double red[33];
  const int pr = group_of(start, nprob, blockIdx.x);
  const GGm& g = tab[pr];
  const int64_t blk = (int64_t)blockIdx.x - start[pr], nb = (int64_t)start[pr + 1] - start[pr];
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (!*g.skip) {
    const int k = g.st->j;
    for (int c = threadIdx.x; c < k; c += blockDim.x) ys[c] = g.y[c];
    __syncthreads();
    for (int64_t i = blk * blockDim.x + threadIdx.x; i < g.m; i += nb * blockDim.x) {
      double acc = 0.0;
      for (int c = 0; c < k; ++c) acc += g.V[(int64_t)c * g.ld + i] * ys[c];
      acc *= g.alpha;
      const double nv = g.r[i] + acc;
      g.r[i] = nv;
      s[0] += acc * acc;
      s[1] += nv * nv;
    }
    for (int64_t i = blk * blockDim.x + threadIdx.x; i < g.n; i += nb * blockDim.x) {
      double acc = 0.0;
      if (g.zb_f32)
        for (int c = 0; c < k; ++c) acc += (double)static_cast<const float*>(g.Zb)[(int64_t)c * g.ldz + i] * ys[c];
      else
        for (int c = 0; c < k; ++c) acc += static_cast<const double*>(g.Zb)[(int64_t)c * g.ldz + i] * ys[c];
      const double nv = g.x[i] + acc;
      g.x[i] = nv;
      s[2] += acc * acc;
      s[3] += nv * nv;
    }
  }
  for (int q = 0; q < 4; ++q) {
    const double v = block_sum_d(s[q], red);
    if (threadIdx.x == 0) g.p4[q * nb + blk] = v;
  }
}

__global__ void grouped_gm_norms_kernel(const GGm* __restrict__ tab, const int* __restrict__ start) {
  __shared__ double red[33];
  const GGm& g = tab[blockIdx.x];
  const int nb = start[blockIdx.x + 1] - start[blockIdx.x];
  for (int q = 0; q < 4; ++q) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += g.p4[q * nb + b];
    s = block_sum_d(s, red);
    if (threadIdx.x == 0) g.nrm[q] = s;
  }
}

cudaError_t launch_grouped_gm_update(const GGm* tab, const int* start, int64_t ctas, int nprob,
                                     cudaStream_t st) {
  if (ctas <= 0) return cudaSuccess;
  const size_t smem = (size_t)kMaxGmresBatch * kMaxGmresBatch * 8;
  cudaError_t e = allow_dyn_smem(grouped_gm_solve_kernel, smem);
  if (e != cudaSuccess) return e;
  grouped_gm_solve_kernel<<<(unsigned)nprob, kGmSolveThreads, smem, st>>>(tab);
  grouped_gm_apply_kernel<<<(unsigned)ctas, 256, 0, st>>>(tab, start, nprob);
  grouped_gm_norms_kernel<<<(unsigned)nprob, 256, 0, st>>>(tab, start);
  return cudaGetLastError();
}

}  // namespace lsq
