// Algorithm 1 (the QR of the sketch): Householder QR of the sketch Y (s x n) in precision
// u_QR (FP32 or FP64), R factor only; the reflectors are also applied to the
// sketched right-hand side (column n), giving c = (Q^T Omega b)[:n] for the
// sketch-and-solve start x_s = R^-1 c (Sec. 4).
//
// Reflector k (Golub & Van Loan): x = W[k:, k], alpha = ||x||, v = x + sign(x_1)
// alpha e_1, H = I - v v^T / (alpha (alpha + |x_1|)); R_kk = -sign(x_1) alpha.
//
// s <= 4096 (and the batch, s <= 1024): column blocks in registers, one launch (qr_block_kernel).
// Longer columns: qr_kernel (FP32) and qr64_kernel (FP64), one cooperative launch of n steps; per step
// every CTA loads v into shared memory and updates whole trailing columns, the one owning column k+1
// also leaves its squared norm for the next step, and a bounded grid barrier separates the steps.
#include <algorithm>
#include <cooperative_groups.h>

#include "common.cuh"
#include "batch.h"
#include "kernels.h"

namespace lsq {

template <typename T>
__device__ __forceinline__ T block_sum_256(T v, T* red) {
  v = warp_sum(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  T t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : T(0);
  if (warp == 0) t = warp_sum(t);
  if (threadIdx.x == 0) red[32] = t;
  __syncthreads();
  return red[32];
}

template <typename T>
__global__ void convert_y_kernel(const double* __restrict__ Y, T* __restrict__ W, int64_t total) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < total) W[i] = (T)Y[i];
}

template <typename T>
__global__ void __launch_bounds__(256) qr_kernel(T* __restrict__ W, int64_t s, int64_t n,
                                                 double* __restrict__ norms,
                                                 double* __restrict__ diagR, unsigned* bar,
                                                 int* err) {
  extern __shared__ __align__(16) unsigned char qr_smem[];
  T* vs = reinterpret_cast<T*>(qr_smem);
  __shared__ T red[33];
  const unsigned nb = gridDim.x;
  if (blockIdx.x == 0) {
    T part = 0;
    for (int64_t t = threadIdx.x; t < s; t += blockDim.x) part += W[t] * W[t];
    const T nn = block_sum_256(part, red);
    if (threadIdx.x == 0) norms[0] = (double)nn;
  }
  if (!grid_barrier(bar, bar + 1, nb, err)) return;
  for (int64_t k = 0; k < n; ++k) {
    const T* colk = W + k * s;
    const T alpha = sqrt((T)norms[k]);
    const T x0 = colk[k];
    const T sgn = (x0 >= T(0)) ? T(1) : T(-1);
    const T scale = (alpha > T(0)) ? T(1) / (alpha * (alpha + fabs(x0))) : T(0);
    if (blockIdx.x == 0 && threadIdx.x == 0) diagR[k] = (double)(-sgn * alpha);
    const int64_t len = s - k;
    for (int64_t t = threadIdx.x; t < len; t += blockDim.x) vs[t] = (t == 0) ? x0 + sgn * alpha : colk[k + t];
    __syncthreads();
    for (int64_t j = k + 1 + blockIdx.x; j <= n; j += nb) {
      T* colj = W + j * s + k;
      T part = 0;
      for (int64_t t = threadIdx.x; t < len; t += blockDim.x) part += vs[t] * colj[t];
      const T wj = block_sum_256(part, red) * scale;
      T part2 = 0;
      for (int64_t t = threadIdx.x; t < len; t += blockDim.x) {
        const T val = colj[t] - wj * vs[t];
        colj[t] = val;
        if (t >= 1) part2 += val * val;
      }
      if (j == k + 1 && j < n) {
        const T nn = block_sum_256(part2, red);
        if (threadIdx.x == 0) norms[k + 1] = (double)nn;
      }
    }
    if (!grid_barrier(bar, bar + 1, nb, err)) return;
  }
}

// FP64 variant (u_QR = double) for GB300's narrow FP64 pipe: one 512-thread CTA per SM.
// Step k: every CTA loads v_k into shared memory; CTA b takes a contiguous share of the
// trailing columns k+1..n (column n is Omega b) and treats them eight at a time: one sweep
// over the rows forms the eight dot products v^T y_j (eight independent FMA chains per
// thread), one reduce-scatter butterfly per warp and sixteen-term sums give w_j, and a
// second sweep applies y_j -= (w_j tau) v (the owner of column k+1 also sums the squares of
// its updated rows 1.. for the next norm).  One bounded grid barrier per step, as before;
// the same reflectors and per-column arithmetic, with blocked sums.
constexpr int kQr64Threads = 512;

__global__ void __launch_bounds__(kQr64Threads, 1)
    qr64_kernel(double* __restrict__ W, int64_t s, int64_t n, double* __restrict__ norms,
                double* __restrict__ diagR, unsigned* bar, int* err) {
  extern __shared__ __align__(16) unsigned char qr_smem[];
  double* vs = reinterpret_cast<double*>(qr_smem);
  __shared__ double red[16 * 9];
  __shared__ double wsum[8];
  __shared__ double nred[17];
  const unsigned nb = gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (blockIdx.x == 0) {
    double part = 0.0;
    for (int64_t t = threadIdx.x; t < s; t += blockDim.x) part = fma(W[t], W[t], part);
    part = warp_sum(part);
    if (lane == 0) nred[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
      double q = 0.0;
      for (int w = 0; w < nw; ++w) q += nred[w];
      norms[0] = q;
    }
  }
  if (!grid_barrier(bar, bar + 1, nb, err)) return;
  for (int64_t k = 0; k < n; ++k) {
    const double* colk = W + k * s;
    const double alpha = sqrt(__ldcg(norms + k));
    const double x0 = __ldcg(colk + k);
    const double sgn = (x0 >= 0.0) ? 1.0 : -1.0;
    const double tau = (alpha > 0.0) ? 1.0 / (alpha * (alpha + fabs(x0))) : 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) diagR[k] = -sgn * alpha;
    const int64_t len = s - k;
    for (int64_t t = threadIdx.x; t < len; t += blockDim.x) vs[t] = (t == 0) ? x0 + sgn * alpha : __ldcg(colk + k + t);
    __syncthreads();
    const int64_t ntr = n - k;                       // trailing columns k+1..n
    const int64_t per = (ntr + nb - 1) / nb;
    const int64_t j0 = k + 1 + (int64_t)blockIdx.x * per, j1 = min(n + 1, j0 + per);
    for (int64_t g = j0; g < j1; g += 8) {
      double d[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) d[q] = 0.0;
      for (int64_t t = threadIdx.x; t < len; t += blockDim.x) {
        const double vt = vs[t];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (g + q < j1) d[q] = fma(vt, __ldcg(W + (g + q) * s + k + t), d[q]);
      }
      const double tot = warp_reduce8(d);
      if ((lane & 3) == 0) red[warp * 9 + ((lane >> 2) & 7)] = tot;
      __syncthreads();
      if (threadIdx.x < 8) {
        double q = 0.0;
        for (int w = 0; w < nw; ++w) q += red[w * 9 + threadIdx.x];
        wsum[threadIdx.x] = q * tau;
      }
      __syncthreads();
      const bool owner = (g == k + 1) && (k + 1 < n);   // column k+1 leaves its norm
      double sq = 0.0;
      for (int64_t t = threadIdx.x; t < len; t += blockDim.x) {
        const double vt = vs[t];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (g + q < j1) {
            double* p = W + (g + q) * s + k + t;
            const double val = fma(-wsum[q], vt, *p);
            *p = val;
            if (q == 0 && owner && t >= 1) sq = fma(val, val, sq);
          }
        }
      }
      if (owner) {
        sq = warp_sum(sq);
        if (lane == 0) nred[warp] = sq;
        __syncthreads();
        if (threadIdx.x == 0) {
          double q = 0.0;
          for (int w = 0; w < nw; ++w) q += nred[w];
          norms[k + 1] = q;
        }
      }
      __syncthreads();
    }
    if (!grid_barrier(bar, bar + 1, nb, err)) return;
  }
}

// R (FP64, col-major, diag >= 0) and c from the factored work matrix.
template <typename T>
__device__ __forceinline__ void qr_finalize_body(const T* __restrict__ W, int64_t s, int64_t n,
                                                 const double* __restrict__ diagR, double* __restrict__ R,
                                                 double* __restrict__ c, int64_t j /* column of R */) {
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const double sg = (diagR[i] < 0.0) ? -1.0 : 1.0;
    double v = 0.0;
    if (i == j) v = diagR[i];
    else if (i < j) v = (double)W[j * s + i];
    if (R) R[j * n + i] = v * sg;
    if (c && j == 0) c[i] = (double)W[n * s + i] * sg;
  }
}

template <typename T>
__global__ void qr_finalize_kernel(const T* __restrict__ W, int64_t s, int64_t n,
                                   const double* __restrict__ diagR, double* __restrict__ R,
                                   double* __restrict__ c) {
  qr_finalize_body<T>(W, s, n, diagR, R, c, blockIdx.x);
}

// ------------------------------------------------------------ register-block variant
// Column blocks of NB, one CTA per block, the block's columns in registers for the whole
// factorization (thread t holds rows t, t + NT, ... of every column); one launch.  CTA q waits
// for the flag of each block P < q in turn, applies its reflectors (compact WY,
// with V, tau and the Gram entries read from global memory), then factors its own block,
// publishes V (below the diagonal of W, R above) and those, and raises its flag; so the next block's chain runs while
// the others still apply.  Column Householder steps take one block reduction each: the dot
// products x_j^T x_c of the pivot column with every column of the block at once (c = j is the
// squared norm), from which v = x_j + sgn alpha e_j gives v^T x_c = x_j^T x_c + sgn alpha x_c[j].  The
// registers rotate by one column a step, so the step is a loop and not NB copies of its
// code; after NB steps every column is back in its place, and the products with finished
// columns are the Gram entries g_lj = v_l^T v_j.  With them the block's reflectors apply as
// w_a = tau_a (v_a^T x - sum_{l < a} g_la w_l), x -= V w (the triangular system of the compact-WY
// form; forming T itself inside the column steps took half of a step's time).
//
// Bound by the chain of the blocks (flag, V from L2, two products, NB column steps).  Panels
// of 16 columns on one CTA of 1024 threads, unrolled over the columns (each launch fetched
// some 10,000 instructions once), two reductions a column, and a launch for each trailing
// update took 1.93 ms at s = 2000, n = 500 in FP32, and a grid barrier per column 1.9 ms at s =
// 748, n = 187 in FP64; now 0.95 and 0.96 ms.  NB: 8 in FP32; 4 in FP64, where a CTA's arithmetic (two FMAs a
// clock an SM) weighs as much as the latency.
constexpr int min_int(int a, int b) { return a < b ? a : b; }
template <typename T, int N>
__device__ __forceinline__ T warp_reduce_scatter(T (&v)[N], int lane) {
  // after the call lane l holds the warp total of v[l / (32 / N)]
  static_assert(N == 4 || N == 8 || N == 16 || N == 32, "a power of two up to the warp");
  int cnt = N;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    if (cnt > 1) {
      const bool upper = (lane & o) != 0;
      const int half = cnt / 2;
#pragma unroll
      for (int t = 0; t < N / 2; ++t) {
        if (t < half) {
          const T send = upper ? v[t] : v[t + half];
          const T keep = upper ? v[t + half] : v[t];
          v[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      cnt = half;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

//
// C > 1: a block's rows are spread over a cluster of C CTAs, so that the chain of a block (in FP64
// a warp issues an instruction in 67 cycles) has C SMs; the partial sums go to every CTA of the
// cluster, one cluster barrier a reduction.  Blocks are taken by ticket (flag[nblk]), so they
// need not all be resident: a block waits only for blocks that run already.  FP64 with the
// columns in shared memory and a flag per column (one SM's FP64 rate bound the pivot column):
// s = 2000, n = 500 5.9 ms, s = 4000, n = 1000 14.8 ms; now 3.1 and 12.3 (5.8 of them FMAs).
// The CTA's (or cluster's) next item.
template <int C>
__device__ __forceinline__ int qr_ticket(unsigned* counter) {
  __shared__ unsigned ticket;
  if constexpr (C > 1) {
    cl_sync();   // the whole cluster runs
    if (cl_rank() == 0 && threadIdx.x == 0) {
      const unsigned k = atomicAdd(counter, 1u);
      for (int d = 0; d < C; ++d) st_cluster(cl_map(smem_u32(&ticket), (uint32_t)d), k);
    }
    cl_sync();
  } else {
    if (threadIdx.x == 0) ticket = atomicAdd(counter, 1u);
    __syncthreads();
  }
  return (int)ticket;
}

// Block q of the factorization of Y; W receives V and R, Tg and flag hold the blocks' factors and flags.
template <typename T, int NB, int NT, int RPT, int C>
__device__ __forceinline__ void qr_block_body(const double* __restrict__ Y, T* __restrict__ W, int64_t s, int64_t n,
                                              double* __restrict__ diagR, T* __restrict__ Tg,
                                              unsigned* __restrict__ flag, int q, int* err) {
  constexpr int NW = NT / 32;
  constexpr int HA = min_int(NB, 32 / NB);   // reflectors at a time in the products
  constexpr int NH = NB / HA;
  constexpr int LB = NB;                            // columns of V loaded at a time
  __shared__ T red[2][NW][NB * NB];
  // Gs: g_la at l + a * NB (l < a), tau_a at a + a * NB
  __shared__ T Ws[NB * NB], Gs[NB * NB], prow[2][NB];
  __shared__ T sc[2], rd[NB];
  extern __shared__ __align__(16) unsigned char qb_smem[];
  T* Vs = reinterpret_cast<T*>(qb_smem);   // [NB][RPT * NT]: the block of reflectors being applied
  // C > 1: the CTAs' shares of the products of a block (by its parity) and of a column (by the
  // column's), and the pivot row
  __shared__ T cw[C > 1 ? 2 : 1][C][NB * NB], cd[C > 1 ? 2 : 1][C][NB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = C > 1 ? (int)cl_rank() : 0;
  // Row i of a thread.  The pieces of NT rows go round the cluster, so that its CTAs keep equal
  // shares while the factored rows grow; FP64 leaves out the pieces that hold none of a
  // reflector's rows.
  auto row = [&](int i) { return (i * C + rank) * NT + tid; };
  auto idle = [&](int i, int64_t first) {
    if constexpr (sizeof(T) == 4) return false;
    else return (int64_t)(i * C + rank + 1) * NT <= first || (int64_t)(i * C + rank) * NT >= s;
  };
  bool live = true;                           // C > 1: no wait has run out
  const int64_t c0 = (int64_t)q * NB;
  const int ncol = (int)min((int64_t)NB, n + 1 - c0);
  T x[RPT][NB];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int64_t r = row(i);
#pragma unroll
    for (int c = 0; c < NB; ++c) x[i][c] = (r < s && c < ncol) ? (T)Y[(c0 + c) * s + r] : T(0);
  }
  // ---- reflectors of the earlier blocks
  for (int P = 0; P < q; ++P) {
    int ok = 1;
    if (tid == 0) {
      const unsigned* fp = flag + P;
      auto raised = [&]() {
        unsigned f;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(fp) : "memory");
        return f >= (unsigned)C;
      };
      if (live && !raised()) {
        const uint64_t t0 = globaltimer_ns();
        while (!raised()) {
          if (globaltimer_ns() - t0 > kWaitLimitNs) {
            set_error(err, DEV_TIMEOUT_GRID);
            ok = 0;
            break;
          }
        }
      }
    }
    if (__syncthreads_and(ok) == 0) {
      if constexpr (C == 1) return;
      else live = false;   // the cluster's barriers need every CTA: go on without waiting
    }
    const int64_t p = (int64_t)P * NB;
    if (tid < NB * NB) Gs[tid] = __ldcg(Tg + (int64_t)P * NB * NB + tid);
    // a thread stages its own rows of V (from L2; zero above each diagonal entry), all loads in
    // flight together where the registers allow it
    const T* V = W + p * s;
#pragma unroll
    for (int a0 = 0; a0 < NB; a0 += LB) {
      T v[LB][RPT];
#pragma unroll
      for (int a = 0; a < LB; ++a)
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          const int64_t r = row(i);
          v[a][i] = (!idle(i, p) && r >= p + a0 + a && r < s) ? __ldcg(V + (a0 + a) * s + r) : T(0);
        }
#pragma unroll
      for (int a = 0; a < LB; ++a)
#pragma unroll
        for (int i = 0; i < RPT; ++i) Vs[(a0 + a) * (RPT * NT) + tid + i * NT] = v[a][i];
    }
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      T acc[HA * NB];
#pragma unroll
      for (int e = 0; e < HA * NB; ++e) acc[e] = T(0);
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        if (!idle(i, p)) {   // V is zero outside its rows
          const int r = tid + i * NT;
          T v[HA];
#pragma unroll
          for (int a = 0; a < HA; ++a) v[a] = Vs[(h * HA + a) * (RPT * NT) + r];
#pragma unroll
          for (int a = 0; a < HA; ++a)
#pragma unroll
            for (int c = 0; c < NB; ++c) acc[a * NB + c] = fma(v[a], x[i][c], acc[a * NB + c]);
        }
      }
      const T w = warp_reduce_scatter<T, HA * NB>(acc, lane);
      constexpr int LP = 32 / (HA * NB);   // lanes per value
      if (lane % LP == 0) red[0][warp][h * HA * NB + lane / LP] = w;
    }
    __syncthreads();
    if constexpr (C == 1) {
      if (tid < NB * NB) {
        T w = T(0);
#pragma unroll
        for (int k = 0; k < NW; ++k) w += red[0][k][tid];
        Ws[tid] = w;
      }
      __syncthreads();
    } else {
      // warp d sends this CTA's share to the CTAs d, d + NW, ...
      for (int e = lane; e < NB * NB; e += 32) {
        T w = T(0);
#pragma unroll
        for (int k = 0; k < NW; ++k) w += red[0][k][e];
        for (int d = warp; d < C; d += NW) st_cluster(cl_map(smem_u32(&cw[P & 1][rank][e]), (uint32_t)d), w);
      }
      cl_sync();
      if (tid < NB * NB) {
        T w = T(0);
#pragma unroll
        for (int d = 0; d < C; ++d) w += cw[P & 1][d][tid];
        Ws[tid] = w;
      }
      __syncthreads();
    }
    if (tid < NB) {   // column tid of the block: forward substitution
      T w[NB];
#pragma unroll
      for (int a = 0; a < NB; ++a) {
        T u = Ws[a * NB + tid];
#pragma unroll
        for (int l = 0; l < a; ++l) u = fma(-Gs[l + a * NB], w[l], u);
        w[a] = Gs[a + a * NB] * u;
        Ws[a * NB + tid] = w[a];
      }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      T w2[HA * NB];
#pragma unroll
      for (int e = 0; e < HA * NB; ++e) w2[e] = Ws[h * HA * NB + e];
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        if (!idle(i, p)) {   // V is zero outside its rows
          const int r = tid + i * NT;
          T v[HA];
#pragma unroll
          for (int a = 0; a < HA; ++a) v[a] = Vs[(h * HA + a) * (RPT * NT) + r];
#pragma unroll
          for (int c = 0; c < NB; ++c) {
            T y = x[i][c];
#pragma unroll
            for (int a = 0; a < HA; ++a) y = fma(-v[a], w2[a * NB + c], y);
            x[i][c] = y;
          }
        }
      }
    }
  }
  // ---- factor the own block
  const int kb = (int)max((int64_t)0, min((int64_t)NB, n - c0));
  if (tid < NB * NB) Gs[tid] = T(0);
  __syncthreads();
#pragma unroll 1
  for (int j = 0; j < NB; ++j) {
    // x[.][c] holds column (j + c) % NB of the block
    if (j < kb) {
      const int pr = (int)c0 + j;
      const int par = j & 1;
      T d[NB];
#pragma unroll
      for (int c = 0; c < NB; ++c) d[c] = T(0);
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = row(i);
        if (idle(i, pr)) continue;
        const T xj = r >= pr ? x[i][0] : T(0);
#pragma unroll
        for (int c = 0; c < NB; ++c) d[c] = fma(xj, x[i][c], d[c]);
        if (r == pr) {
#pragma unroll
          for (int c = 0; c < NB; ++c) {
            if constexpr (C == 1) {
              prow[par][c] = x[i][c];
            } else {
              for (int d = 0; d < C; ++d) st_cluster(cl_map(smem_u32(&prow[par][c]), (uint32_t)d), x[i][c]);
            }
          }
        }
      }
      const T dw = warp_reduce_scatter<T, NB>(d, lane);
      constexpr int LP = 32 / NB;
      if (lane % LP == 0) red[par][warp][lane / LP] = dw;
      __syncthreads();
      if constexpr (C > 1) {
        // a CTA's share by lanes 0 .. NB - 1 of each warp, which sends it to the CTAs warp, warp + NW, ...
        if (lane < NB) {
          T w = T(0);
#pragma unroll
          for (int k = 0; k < NW; ++k) w += red[par][k][lane];
          for (int d = warp; d < C; d += NW) st_cluster(cl_map(smem_u32(&cd[par][rank][lane]), (uint32_t)d), w);
        }
        cl_sync();
      }
      T tot = T(0), sa, tau;   // lane l: value l % NB, summed over a share of the warps, then over the shares
      const T x0 = prow[par][0];
      auto totals = [&]() {
#pragma unroll
        for (int k = 0; k < ((C > 1 ? C : NW) + LP - 1) / LP; ++k)
          if (lane / NB + k * LP < (C > 1 ? C : NW)) {
            if constexpr (C > 1) tot += cd[par][lane / NB + k * LP][lane % NB];
            else tot += red[par][lane / NB + k * LP][lane % NB];
          }
#pragma unroll
        for (int o = NB; o < 32; o <<= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      };
      auto scalars = [&](T n2) {
        const T alpha = sqrt(n2);
        sa = (x0 >= T(0)) ? alpha : -alpha;
        tau = (alpha > T(0)) ? T(1) / (alpha * (alpha + fabs(x0))) : T(0);
      };
      if constexpr (sizeof(T) == 4) {
        totals();
        scalars(__shfl_sync(0xffffffffu, tot, 0));
      } else {   // FP64 is scarce: the sums, the root and the quotient in one warp
        if (warp == 0) {
          totals();
          scalars(__shfl_sync(0xffffffffu, tot, 0));
          if (lane < NB) red[par][0][lane] = tot;   // every warp's share has been read by this warp alone
          if (lane == 0) {
            sc[0] = sa;
            sc[1] = tau;
          }
        }
        __syncthreads();
        tot = red[par][0][lane % NB];
        sa = sc[0];
        tau = sc[1];
      }
      T v[RPT];   // v_j: zero above the pivot row, where x keeps R
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int r = row(i);
        if (r == pr) x[i][0] += sa;
        v[i] = r >= pr ? x[i][0] : T(0);
        // the column is final: R above the pivot row, v_j from it down
        if (r < s) W[(int64_t)pr * s + r] = x[i][0];
      }
#pragma unroll
      for (int c = 1; c < NB; ++c) {
        const T vx = fma(sa, prow[par][c], __shfl_sync(0xffffffffu, tot, c));
        if (c < NB - j) {
          const T coef = tau * vx;
#pragma unroll
          for (int i = 0; i < RPT; ++i)
            if (!idle(i, pr)) x[i][c] = fma(-coef, v[i], x[i][c]);
        }
      }
      if (warp == 0) {   // lane c >= NB - j: v_l^T v_j of the finished column l = c - (NB - j)
        if (lane < NB && lane >= NB - j) Gs[lane - (NB - j) + j * NB] = fma(sa, prow[par][lane], tot);
        if (lane == 0) {
          Gs[j + j * NB] = tau;
          rd[j] = -sa;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const T first = x[i][0];
#pragma unroll
      for (int c = 0; c + 1 < NB; ++c) x[i][c] = x[i][c + 1];
      x[i][NB - 1] = first;
    }
  }
  // ---- the right-hand side's column, if the block holds it; tau and the Gram entries; the flag
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int64_t r = row(i);
#pragma unroll
    for (int c = 0; c < NB; ++c)
      if (c >= kb && c < ncol && r < s) W[(c0 + c) * s + r] = x[i][c];
  }
  __syncthreads();
  if (rank == 0) {
    if (tid < NB * NB) Tg[(int64_t)q * NB * NB + tid] = Gs[tid];
    if (tid < kb) diagR[c0 + tid] = (double)rd[tid];
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) atomicAdd(flag + q, 1u);
  if constexpr (C > 1) cl_sync();   // no CTA leaves while another may still send to it
}

template <typename T, int NB, int NT, int RPT, int C>
__global__ void __launch_bounds__(NT, 1)
    qr_block_kernel(const double* __restrict__ Y, T* __restrict__ W, int64_t s, int64_t n, double* __restrict__ diagR,
                    T* __restrict__ Tg, unsigned* __restrict__ flag, int nblk, int* err) {
  const int q = C > 1 ? qr_ticket<C>(flag + nblk) : (int)blockIdx.x;
  qr_block_body<T, NB, NT, RPT, C>(Y, W, s, n, diagR, Tg, flag, q, err);
}

// The register-block form: `aux` as launch_qr's, block factors and flags behind diag(R).
template <typename T, int NB, int NT, int RPT, int C = 1>
static cudaError_t run_qr_block(const double* Y, int64_t s, int64_t n, T* W, double* aux, double* R, double* c,
                                int* err, cudaStream_t st) {
  const unsigned nblk = (unsigned)((n + 1 + NB - 1) / NB);
  double* diagR = aux + n;
  T* Tg = reinterpret_cast<T*>(aux + 2 * n + 8);
  unsigned* flag = reinterpret_cast<unsigned*>(Tg + (size_t)nblk * NB * NB);
  cudaError_t e = cudaMemsetAsync(flag, 0, (nblk + 1) * sizeof(unsigned), st);   // and the ticket
  if (e != cudaSuccess) return e;
  T* Wp = W;
  int64_t sp = s, np = n;
  int nb = (int)nblk;
  size_t smem = (size_t)NB * RPT * NT * sizeof(T);
  // at most three CTAs an SM: with more, the FP64 instructions of the block that all others wait
  // for queue behind theirs (s = 4000, n = 1000: 13.2 ms with four, 12.3 with three, 17 with two;
  // without the limit / with it, ms: s = 2000, n = 500 3.48 / 3.15, 1000 x 250 1.30 / 1.26, 500 x 125 and
  // FP32 the same)
  if (C > 1) smem = std::max(smem, (size_t)74 * 1024);
  auto kern = qr_block_kernel<T, NB, NT, RPT, C>;
  e = allow_dyn_smem(kern, smem);
  if (e != cudaSuccess) return e;
  if constexpr (C == 1) {
    void* args[] = {&Y, &Wp, &sp, &np, &diagR, &Tg, &flag, &nb, &err};
    e = cudaLaunchCooperativeKernel((const void*)kern, dim3(nblk), dim3(NT), args, smem, st);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk * C);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, Y, Wp, sp, np, diagR, Tg, flag, nb, err);
  }
  if (e != cudaSuccess) return e;
  qr_finalize_kernel<T><<<(unsigned)n, 256, 0, st>>>(W, s, n, diagR, R, c);
  return cudaGetLastError();
}

// Bytes of the region behind diag(R) in aux that a factorization of n columns may use.
size_t qr_aux_tail(int64_t n) {
  const size_t f32 = (size_t)((n + 1 + 7) / 8) * (64 * 4 + 4) + 4, f64 = (size_t)((n + 1 + 3) / 4) * (16 * 8 + 4) + 4;
  return std::max(f32, f64);
}

template <typename T>
static cudaError_t run_qr(const double* Y, int64_t s, int64_t n, T* W, double* aux, unsigned* bar,
                          double* R, double* c, int* err, int num_sms, cudaStream_t st) {
  const int64_t total = s * (n + 1);
  convert_y_kernel<T><<<(unsigned)((total + 255) / 256), 256, 0, st>>>(Y, W, total);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)s * sizeof(T);
  auto kern = qr_kernel<T>;
  if (smem > 48 * 1024) {
    e = allow_dyn_smem(kern, smem);
    if (e != cudaSuccess) return e;
  }
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 256, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  int64_t grid = (int64_t)occ * num_sms;
  if (grid > n) grid = n;
  if (grid < 1) grid = 1;
  double* norms = aux;
  double* diagR = aux + n;
  T* Wp = W;
  int64_t sp = s, np = n;
  void* args[] = {&Wp, &sp, &np, &norms, &diagR, &bar, &err};
  e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)grid), dim3(256), args, smem, st);
  if (e != cudaSuccess) return e;
  qr_finalize_kernel<T><<<(unsigned)n, 256, 0, st>>>(W, s, n, diagR, R, c);
  return cudaGetLastError();
}

static cudaError_t run_qr64(const double* Y, int64_t s, int64_t n, double* W, double* aux, unsigned* bar,
                           double* R, double* c, int* err, int num_sms, cudaStream_t st) {
  const int64_t total = s * (n + 1);
  cudaError_t e = cudaMemcpyAsync(W, Y, (size_t)total * 8, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const int grid = num_sms;                      // one CTA per SM (co-resident: occ >= 1)
  const size_t smem = (size_t)s * 8;
  e = allow_dyn_smem(qr64_kernel, smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, qr64_kernel, kQr64Threads, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  double* norms = aux;
  double* diagR = aux + n;
  double* Wp = W;
  int64_t sp = s, np = n;
  void* args[] = {&Wp, &sp, &np, &norms, &diagR, &bar, &err};
  e = cudaLaunchCooperativeKernel((const void*)qr64_kernel, dim3((unsigned)grid), dim3(kQr64Threads), args, smem, st);
  if (e != cudaSuccess) return e;
  qr_finalize_kernel<double><<<(unsigned)n, 256, 0, st>>>(W, s, n, diagR, R, c);
  return cudaGetLastError();
}

cudaError_t launch_qr(bool fp64, const double* Y, int64_t s, int64_t n, void* work, double* aux,
                      unsigned* bar, double* R, double* c, int* err, int num_sms, cudaStream_t st) {
  if (!fp64) {
    float* W = static_cast<float*>(work);
    // one CTA per block of eight columns, all co-resident (n <= 1024: at most 129), rows of a
    // column in at most eight registers of each thread
    if ((n + 1 + 7) / 8 <= num_sms) {
      if (s <= 512) return run_qr_block<float, 8, 256, 2>(Y, s, n, W, aux, R, c, err, st);
      if (s <= 1024) return run_qr_block<float, 8, 256, 4>(Y, s, n, W, aux, R, c, err, st);
      if (s <= 2048) return run_qr_block<float, 8, 256, 8>(Y, s, n, W, aux, R, c, err, st);
    }
    // past that a cluster of eight (s = 4000, n = 1000: 2.94 ms with 512 threads of eight rows on one
    // CTA, 2.06 so; at s <= 2048 the cluster's barriers cost more than they give: 0.94 and 0.96)
    if (s > 2048 && s <= 4096) return run_qr_block<float, 8, 256, 2, 8>(Y, s, n, W, aux, R, c, err, st);
    return run_qr<float>(Y, s, n, W, aux, bar, R, c, err, num_sms, st);
  }
  double* W = static_cast<double*>(work);
  // FP64: rows of a block over clusters of four or eight CTAs, fewer rows a thread than a
  // wider CTA would have (s = 1000, n = 250: 1.81 ms on one CTA of 128 threads, 1.24 so)
  if (s <= 256) return run_qr_block<double, 4, 64, 1, 4>(Y, s, n, W, aux, R, c, err, st);
  if (s <= 512) return run_qr_block<double, 4, 128, 1, 4>(Y, s, n, W, aux, R, c, err, st);
  if (s <= 1024) return run_qr_block<double, 4, 64, 2, 8>(Y, s, n, W, aux, R, c, err, st);
  if (s <= 2048) return run_qr_block<double, 4, 64, 4, 8>(Y, s, n, W, aux, R, c, err, st);
  if (s <= 4096) return run_qr_block<double, 4, 128, 4, 8>(Y, s, n, W, aux, R, c, err, st);
  return run_qr64(Y, s, n, W, aux, bar, R, c, err, num_sms, st);
}


// ============================================================ grouped (batched) QR
// The register-block form for all problems in one launch (s <= 1024): the blocks of problem p
// are items start[p] .. start[p + 1] - 1, taken by ticket, so an item waits only for items that run
// already.  One CTA of 1024 threads per problem, with W in global memory, took as long as its
// largest problem's chain (n = 256, s = 1024: 4.2 ms; 0.50 now for a batch of 32).
template <typename T, int NB, int NT, int RPT, int C>
__global__ void __launch_bounds__(NT, 1)
    grouped_qr_kernel(const GQr<T>* __restrict__ tab, const int* __restrict__ start, int nprob, T* __restrict__ Tg,
                      unsigned* __restrict__ flag, int* err) {
  const int t = qr_ticket<C>(flag + start[nprob]);
  const int p = group_of(start, nprob, t);
  const GQr<T> g = tab[p];
  qr_block_body<T, NB, NT, RPT, C>(g.Y, g.W, g.s, g.n, g.diagR, Tg + (int64_t)start[p] * NB * NB, flag + start[p],
                                   t - start[p], err);
}

template <typename T, int NB, int NT, int RPT, int C>
static cudaError_t run_grouped_qr(const GQr<T>* tab, const int* start, int64_t blocks, int nprob, void* work, int* err,
                                  cudaStream_t st) {
  T* Tg = static_cast<T*>(work);
  unsigned* flag = reinterpret_cast<unsigned*>(Tg + (size_t)blocks * NB * NB);
  cudaError_t e = cudaMemsetAsync(flag, 0, (blocks + 1) * sizeof(unsigned), st);   // and the ticket
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)NB * RPT * NT * sizeof(T);
  auto kern = grouped_qr_kernel<T, NB, NT, RPT, C>;
  e = allow_dyn_smem(kern, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(blocks * C));
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, tab, start, nprob, Tg, flag, err);
}

template <typename T>
__global__ void grouped_qr_finalize_kernel(const GQr<T>* __restrict__ tab, const int* __restrict__ start, int nprob) {
  const int p = group_of(start, nprob, blockIdx.x);
  const GQr<T>& g = tab[p];
  qr_finalize_body<T>(g.W, g.s, g.n, g.diagR, g.R, g.c, (int64_t)blockIdx.x - start[p]);
}

template <typename T>
cudaError_t launch_grouped_qr(const GQr<T>* tab, const int* blk_start, int64_t blocks, const int* col_start,
                              int64_t col_ctas, int nprob, int64_t max_s, void* work, int* err, cudaStream_t st) {
  if (nprob <= 0) return cudaSuccess;
  if (max_s > 1024) return cudaErrorInvalidValue;
  cudaError_t e;
  // the two forms of a type differ in the rows a thread holds alone: to a problem with s <= 512 the
  // longer form adds rows of zeros, so its bits do not depend on the batch's largest s
  if constexpr (sizeof(T) == 4)
    e = max_s <= 512 ? run_grouped_qr<T, 8, 256, 2, 1>(tab, blk_start, blocks, nprob, work, err, st)
                     : run_grouped_qr<T, 8, 256, 4, 1>(tab, blk_start, blocks, nprob, work, err, st);
  else
    e = max_s <= 512 ? run_grouped_qr<T, 4, 128, 1, 4>(tab, blk_start, blocks, nprob, work, err, st)
                     : run_grouped_qr<T, 4, 128, 2, 4>(tab, blk_start, blocks, nprob, work, err, st);
  if (e != cudaSuccess) return e;
  grouped_qr_finalize_kernel<T><<<(unsigned)col_ctas, 256, 0, st>>>(tab, col_start, nprob);
  return cudaGetLastError();
}
template cudaError_t launch_grouped_qr<float>(const GQr<float>*, const int*, int64_t, const int*, int64_t, int, int64_t, void*,
                                              int*, cudaStream_t);
template cudaError_t launch_grouped_qr<double>(const GQr<double>*, const int*, int64_t, const int*, int64_t, int, int64_t,
                                               void*, int*, cudaStream_t);

}  // namespace lsq
