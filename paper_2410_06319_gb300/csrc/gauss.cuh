// The sketch matrix G of Omega = s^-1/2 fl_s(G), generated on the fly.
//
// Definition (Sec. 2 Gaussian embedding with N(0, 1/s) entries; Sec. 5 uses
// Omega = (4n)^-1/2 G): G[i, j] for sketch row i and data row j is
//   (x0, x1, x2, x3) = Philox4x32-10(counter = (j>>2, i, j>>34, 0),
//                                    key = (seed lo, seed hi))        [SC'11]
//   (a, b) = (x0, x1) if j%4 < 2 else (x2, x3)
//   U1 = (a + 1) 2^-32,  U2 = b 2^-32,  R = sqrt(-2 ln U1)
//   G = R cos(2 pi U2) for even j, R sin(2 pi U2) for odd j; G = +0 if a = 2^32-1
// with ln and (cos, sin)(2 pi U2) evaluated by the fixed IEEE double sequences
// spec_ln_u1 / spec_cos_sin_2pi below (no fused multiply-add).  The operand
// used by a sketch in precision u_s is fl_s(G), round to nearest even.
//
// Evaluation on GB300: FP64 is a slow pipe, so G is first estimated in FP32 with a bound on
// the error (gauss_pair_est).  Where the whole interval rounds to one u_s value, that value
// is fl_s(G) exactly.  The other pairs are evaluated in double-float (two FP32 words) and, in
// the rare case that this does not decide them either, by the FP64 definition, rounded once
// (round to odd into FP32, then to u_s).  The result is bit-identical to rounding the FP64
// definition directly.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

namespace lsq {

enum SFmt : int { FMT_F64 = 0, FMT_F32 = 1, FMT_F16 = 2, FMT_BF16 = 3, FMT_E4M3 = 4, FMT_BF16X3 = 5 };

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // one 32 x 32 -> 64 bit product each
    const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k0, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k1, (uint32_t)p0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// Counter of the Philox call serving sketch row i, data rows 4q .. 4q+3.
__device__ __forceinline__ uint4 gauss_counter(uint64_t q, uint32_t i) {
  return make_uint4((uint32_t)q, i, (uint32_t)(q >> 32), 0u);
}

// ------------------------------------------------------------ FP64 definition
__device__ __forceinline__ double spec_ln_u1(uint32_t a) {
  // U1 = 2^e f, f in [sqrt(1/2), sqrt(2)); ln f = 2 atanh(z), z = (f-1)/(f+1),
  // series 2z (1 + w/3 + ... + w^11/23), w = z^2, Horner with separate * and +.
  const double u1 = (double)((uint64_t)a + 1ull) * 0x1p-32;
  const long long bits = __double_as_longlong(u1);
  double e = (double)((int)((bits >> 52) & 0x7FF) - 1023);
  double f = __longlong_as_double((bits & 0x000FFFFFFFFFFFFFLL) | 0x3FF0000000000000LL);
  if (f > 1.4142135623730951) {
    f = __dmul_rn(f, 0.5);
    e = __dadd_rn(e, 1.0);
  }
  const double z = __ddiv_rn(__dsub_rn(f, 1.0), __dadd_rn(f, 1.0));
  const double w = __dmul_rn(z, z);
  double p = 1.0 / 23.0;
  p = __dadd_rn(1.0 / 21.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 19.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 17.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 15.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 13.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 11.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 9.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 7.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 5.0, __dmul_rn(w, p));
  p = __dadd_rn(1.0 / 3.0, __dmul_rn(w, p));
  const double z2 = __dmul_rn(z, 2.0);
  const double lnf = __dadd_rn(z2, __dmul_rn(z2, __dmul_rn(w, p)));
  return __dadd_rn(__dmul_rn(e, 0.6931471805599453), lnf);
}

__device__ __forceinline__ void spec_cos_sin_2pi(uint32_t b, double& c, double& s) {
  // 4 U2 = q + r, r moved to [-1/2, 1/2); phi = r (pi/2); Taylor series of sin
  // and cos to phi^21 / phi^20 (Horner, separate * and +); rotate by q.
  uint32_t q = b >> 30;
  int32_t rb = (int32_t)(b & 0x3FFFFFFFu);
  if (rb >= (1 << 29)) {
    rb -= (1 << 30);
    q = (q + 1u) & 3u;
  }
  const double r = (double)rb * 0x1p-30;
  const double phi = __dmul_rn(r, 1.5707963267948966);
  const double w = __dmul_rn(phi, phi);
  double ps = 1.0 / 51090942171709440000.0;           // +1/21!
  ps = __dadd_rn(-1.0 / 121645100408832000.0, __dmul_rn(w, ps));
  ps = __dadd_rn(1.0 / 355687428096000.0, __dmul_rn(w, ps));
  ps = __dadd_rn(-1.0 / 1307674368000.0, __dmul_rn(w, ps));
  ps = __dadd_rn(1.0 / 6227020800.0, __dmul_rn(w, ps));
  ps = __dadd_rn(-1.0 / 39916800.0, __dmul_rn(w, ps));
  ps = __dadd_rn(1.0 / 362880.0, __dmul_rn(w, ps));
  ps = __dadd_rn(-1.0 / 5040.0, __dmul_rn(w, ps));
  ps = __dadd_rn(1.0 / 120.0, __dmul_rn(w, ps));
  ps = __dadd_rn(-1.0 / 6.0, __dmul_rn(w, ps));
  const double sphi = __dadd_rn(phi, __dmul_rn(phi, __dmul_rn(w, ps)));
  double pc = 1.0 / 2432902008176640000.0;            // +1/20!
  pc = __dadd_rn(-1.0 / 6402373705728000.0, __dmul_rn(w, pc));
  pc = __dadd_rn(1.0 / 20922789888000.0, __dmul_rn(w, pc));
  pc = __dadd_rn(-1.0 / 87178291200.0, __dmul_rn(w, pc));
  pc = __dadd_rn(1.0 / 479001600.0, __dmul_rn(w, pc));
  pc = __dadd_rn(-1.0 / 3628800.0, __dmul_rn(w, pc));
  pc = __dadd_rn(1.0 / 40320.0, __dmul_rn(w, pc));
  pc = __dadd_rn(-1.0 / 720.0, __dmul_rn(w, pc));
  pc = __dadd_rn(1.0 / 24.0, __dmul_rn(w, pc));
  pc = __dadd_rn(-1.0 / 2.0, __dmul_rn(w, pc));
  const double cphi = __dadd_rn(1.0, __dmul_rn(w, pc));
  switch (q) {
    case 0: c = cphi; s = sphi; break;
    case 1: c = -sphi; s = cphi; break;
    case 2: c = -cphi; s = -sphi; break;
    default: c = sphi; s = -cphi; break;
  }
}

__device__ __forceinline__ void spec_gauss_pair(uint32_t a, uint32_t b, double& ge, double& go) {
  if (a == 0xFFFFFFFFu) {
    ge = 0.0;
    go = 0.0;
    return;
  }
  const double rad = __dsqrt_rn(__dmul_rn(-2.0, spec_ln_u1(a)));
  double c, s;
  spec_cos_sin_2pi(b, c, s);
  ge = __dmul_rn(rad, c);
  go = __dmul_rn(rad, s);
}

// ------------------------------------------------------------ FP32 estimate
// g is estimated in FP32 with a bound d on |g32 - g| (absolute, first order in the
// documented errors of the approximate functions); where both ends of [g32 - d, g32 + d]
// round to the same u_s value, that value is fl_s(G) exactly (rounding is monotone).
// Otherwise the pair goes to the double-float evaluation below.
//
// Cost: the estimate runs once per pair of entries and bounds every sketch (Philox, 21
// instructions a pair, plus this).  The earlier estimate (ln by a quotient and a series,
// sin and cos by quadrant and series, a 2^-19 relative bound, integer rounding tests) took
// 176 issued instructions a pair in all; the approximate functions take about 60.
//
// Errors, U = U1: the conversion of U rounds once (2^-24); lg2.approx: 2^-22 absolute in
// (1/2, 2), 2^-22 relative below; rsqrt.approx: 2^-22.9 relative.  So |rad2 - rad2_exact|
// <= 4.5e-7 + 4e-7 rad2, and |sqrt(x) - sqrt(y)| <= |x - y| / sqrt(x) for x, y > 0 makes that
// |rad - rad_exact| <= 4.5e-7 / rad + 4e-7 rad at any rad; rad2 is kept above 2^-22, where
// d > rad and no sign of g passes the test.
//  * BF16, E4M3 (coarse): sin.approx and cos.approx, 2^-20.5 absolute, on an angle from the
//    23 leading bits of U2 (centred: 2^-21.3, plus 2^-22.2 of roundings):
//    d = 2e-6 rad + 5e-7 / rad, against a first-order sum of 1.8e-6 rad + 4.5e-7 / rad.
//    About 1.4 % of the BF16 pairs and 0.06 % of the E4M3 pairs are left undecided.
//  * F16 (three more bits): sin and cos by quadrant reduction on the exact integer and a short
//    series, 4e-7 relative, so that small entries keep their relative accuracy:
//    d = |g| (1.2e-6 + 5e-7 / rad2), against 1.1e-6 + 4.5e-7 / rad2; about 1.7 % of the pairs
//    are left undecided (8 % with the approximate functions).
__device__ __forceinline__ float mufu_lg2(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float mufu_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float mufu_sin(float x) {
  float r;
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float mufu_cos(float x) {
  float r;
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The halves of x as 2^23 + x >> 16 and 2^23 + (x & 0xFFFF): integer -> FP32 by byte permutes
// (on GB300 the conversion instructions share the narrow FP64 pipe).
__device__ __forceinline__ float half_hi(uint32_t x) { return __uint_as_float(__byte_perm(x, 0x4B000000u, 0x7632)); }
__device__ __forceinline__ float half_lo(uint32_t x) { return __uint_as_float(__byte_perm(x, 0x4B000000u, 0x7610)); }

// Two FP32 values rounded to u_s (nearest even) and packed, the first in the low bits.
template <int FMT>
__device__ __forceinline__ uint32_t pack2(float e, float o) {
  if constexpr (FMT == FMT_F16) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(o), "f"(e));
    return r;
  } else if constexpr (FMT == FMT_BF16) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(o), "f"(e));
    return r;
  } else {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(o), "f"(e));
    return r;
  }
}

// Both entries of one (a, b) word pair, packed; false when they are not decided by the estimate.
template <int FMT>
__device__ __forceinline__ bool gauss_pair_est(uint32_t a, uint32_t b, uint32_t& packed) {
  // U = (a + 1) 2^-32: both products exact, one rounding in the sum
  const float U = fmaf(half_hi(a), 0x1p-16f, -0x1p7f) + fmaf(half_lo(a), 0x1p-32f, -(0x1p-9f - 0x1p-32f));
  const float rad2 = fmaxf(mufu_lg2(U) * -1.3862943611198906f, 0x1p-22f);
  const float irad = mufu_rsqrt(rad2);
  if constexpr (FMT == FMT_F16) {
    const float rad = rad2 * irad;
    // quadrant of U2 (nearest) and the signed remainder, |x| <= 2^31, x 2^-32 quarter turns
    const uint32_t q = (b + 0x20000000u) >> 30;
    const uint32_t y = (b << 2) ^ 0x80000000u;
    const float x = fmaf(half_hi(y), 65536.0f, -(0x1p39f + 0x1p31f)) + (half_lo(y) - 0x1p23f);
    const float phi = x * (float)(1.57079632679489662 * 0x1p-32);
    const float w = phi * phi;
    float ps = 1.0f / 362880.0f;
    ps = fmaf(w, ps, -1.0f / 5040.0f);
    ps = fmaf(w, ps, 1.0f / 120.0f);
    ps = fmaf(w, ps, -1.0f / 6.0f);
    const float sp = fmaf(phi * w, ps, phi);
    float pc = 1.0f / 40320.0f;
    pc = fmaf(w, pc, -1.0f / 720.0f);
    pc = fmaf(w, pc, 1.0f / 24.0f);
    pc = fmaf(w, pc, -0.5f);
    const float cp = fmaf(w, pc, 1.0f);
    const bool swap = (q & 1u) != 0;
    const uint32_t cb = __float_as_uint(swap ? sp : cp) ^ (((q + 1u) & 2u) << 30);
    const uint32_t sb = __float_as_uint(swap ? cp : sp) ^ ((q & 2u) << 30);
    const float ge = rad * __uint_as_float(cb), go = rad * __uint_as_float(sb);
    const float t = fmaf(irad * irad, 5e-7f, 1.2e-6f);
    packed = pack2<FMT>(fmaf(ge, -t, ge), fmaf(go, -t, go));
    return packed == pack2<FMT>(fmaf(ge, t, ge), fmaf(go, t, go));
  } else {
    // (0x7F : b) >> 9 is the pattern of 1 + floor(b / 2^9) 2^-23; minus 3/2 it is U2 - 1/2, which
    // turns the angle by half a turn: (cos, sin)(2 pi U2) = -(cos, sin)(theta), |theta| <= pi
    const float u = __uint_as_float(__funnelshift_r(b, 0x7Fu, 9)) - 1.5f;
    const float th = fmaf(u, 6.28318530717958648f, (float)(6.28318530717958648 * 0x1p-24));
    const float nrad = -rad2 * irad;
    const float ge = nrad * mufu_cos(th), go = nrad * mufu_sin(th);
    const float d = fmaf(nrad, -2e-6f, irad * 5e-7f);
    packed = pack2<FMT>(ge - d, go - d);
    return packed == pack2<FMT>(ge + d, go + d);
  }
}

// ------------------------------------------------------------ double-float evaluation
// The undecided pairs: the definition's value in double-float (an unevaluated sum of two
// FP32 numbers) on the FP32 pipe, about 250 instructions a pair against ~95 FP64 operations
// (64 cycles of a quarter of the SM each).  Relative error of an entry: each
// product, quotient and sum below 2^-43; the FP32 tails of the series enter scaled by at
// most 2.6e-5 (ln), 4e-7 (sin) and 3.7e-6 (cos) times 2^-23: below 2^-38 in all.  An entry
// further than kDfRel = 2^-36 from a rounding boundary of u_s is decided; the rest (about
// 2^-26 of the undecided ones) take the FP64 definition.
constexpr float kDfRel = 0x1p-36f;
struct F2 {
  float h, l;
};
__host__ __device__ constexpr F2 f2c(double v) { return F2{(float)v, (float)(v - (double)(float)v)}; }
__device__ __forceinline__ F2 f2_quick(float a, float b) {   // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return F2{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 f2_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const F2 s = f2_sum(a.h, b.h);
  return f2_quick(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return f2_quick(p, e);
}
__device__ __forceinline__ F2 f2_div(F2 a, F2 b) {
  const float q = __fdividef(a.h, b.h);
  const float p = __fmul_rn(q, b.h);
  float r = __fsub_rn(__fsub_rn(a.h, p), __fmaf_rn(q, b.h, -p));
  r = __fadd_rn(r, __fmaf_rn(-q, b.l, a.l));
  return f2_quick(q, __fdividef(r, b.h));
}
// x < 2^32 as an exact double-float, times `scale` (a power of two)
__device__ __forceinline__ F2 f2_u32(uint32_t x, float scale) {
  const F2 v = f2_quick(__fmaf_rn(half_hi(x), 65536.0f, -0x1p39f), __fsub_rn(half_lo(x), 0x1p23f));
  return F2{__fmul_rn(v.h, scale), __fmul_rn(v.l, scale)};
}

__device__ __forceinline__ F2 df_ln_u1(uint32_t a) {
  F2 num, den;
  float e = 0.0f;
  if (a >= 0xB504F334u) {   // U1 > sqrt(1/2): z = -V / (2 - V), V = 1 - U1
    const F2 V = f2_u32(~a, 0x1p-32f);
    num = F2{-V.h, -V.l};
    den = f2_add(F2{2.0f, 0.0f}, num);
  } else {
    const F2 u = f2_u32(a + 1u, 0x1p-32f);
    const uint32_t E = __float_as_uint(u.h) >> 23;   // 95 .. 126
    e = __uint_as_float(0x4B000000u | E) - (8388608.0f + 127.0f);
    float sc = __uint_as_float((254u - E) << 23);   // 2^-(E - 127)
    if (u.h * sc > 1.41421356f) {
      sc *= 0.5f;
      e += 1.0f;
    }
    const F2 f{u.h * sc, u.l * sc};
    num = f2_add(f, F2{-1.0f, 0.0f});
    den = f2_add(f, F2{1.0f, 0.0f});
  }
  const F2 z = f2_div(num, den);
  const F2 w = f2_mul(z, z);
  float p = 1.0f / 17.0f;
  p = __fmaf_rn(w.h, p, 1.0f / 15.0f);
  p = __fmaf_rn(w.h, p, 1.0f / 13.0f);
  p = __fmaf_rn(w.h, p, 1.0f / 11.0f);
  p = __fmaf_rn(w.h, p, 1.0f / 9.0f);
  p = __fmaf_rn(w.h, p, 1.0f / 7.0f);
  constexpr F2 c5 = f2c(1.0 / 5.0), c3 = f2c(1.0 / 3.0), ln2 = f2c(0.6931471805599453);
  F2 s = f2_add(c5, F2{__fmul_rn(w.h, p), 0.0f});
  s = f2_add(c3, f2_mul(w, s));
  s = f2_mul(w, s);
  const F2 z2{2.0f * z.h, 2.0f * z.l};
  const F2 lnf = f2_add(z2, f2_mul(z2, s));
  return f2_add(f2_mul(F2{e, 0.0f}, ln2), lnf);
}

__device__ __forceinline__ void df_gauss_pair(uint32_t a, uint32_t b, F2& ge, F2& go) {
  const F2 ln = df_ln_u1(a);
  const F2 r2{-2.0f * ln.h, -2.0f * ln.l};
  const float y = mufu_rsqrt(r2.h), s0 = __fmul_rn(r2.h, y);
  const float res = __fadd_rn(-__fmaf_rn(s0, s0, -r2.h), r2.l);
  const F2 rad = f2_quick(s0, __fmul_rn(__fmul_rn(0.5f, y), res));
  // quadrant and signed remainder of 4 U2, as in the estimate
  const uint32_t q = (b + 0x20000000u) >> 30;
  const int32_t x = (int32_t)(b << 2);
  const uint32_t sg = (uint32_t)x & 0x80000000u;
  constexpr F2 pio2 = f2c(1.57079632679489662);
  const F2 phi = f2_mul(f2_u32(x < 0 ? 0u - (uint32_t)x : (uint32_t)x, 0x1p-32f), pio2);   // |phi|
  const F2 w = f2_mul(phi, phi);
  constexpr F2 s7 = f2c(-1.0 / 5040.0), s5 = f2c(1.0 / 120.0), s3 = f2c(-1.0 / 6.0);
  float ps = 1.0f / 6227020800.0f;
  ps = __fmaf_rn(w.h, ps, -1.0f / 39916800.0f);
  ps = __fmaf_rn(w.h, ps, 1.0f / 362880.0f);
  F2 t = f2_add(s7, F2{__fmul_rn(w.h, ps), 0.0f});
  t = f2_add(s5, f2_mul(w, t));
  t = f2_add(s3, f2_mul(w, t));
  const F2 sp = f2_add(phi, f2_mul(phi, f2_mul(w, t)));
  constexpr F2 c6 = f2c(-1.0 / 720.0), c4 = f2c(1.0 / 24.0);
  float pc = 1.0f / 479001600.0f;
  pc = __fmaf_rn(w.h, pc, -1.0f / 3628800.0f);
  pc = __fmaf_rn(w.h, pc, 1.0f / 40320.0f);
  t = f2_add(c6, F2{__fmul_rn(w.h, pc), 0.0f});
  t = f2_add(c4, f2_mul(w, t));
  t = f2_add(F2{-0.5f, 0.0f}, f2_mul(w, t));
  const F2 cp = f2_add(F2{1.0f, 0.0f}, f2_mul(w, t));
  const bool swap = (q & 1u) != 0;
  const uint32_t ssp = sg;   // sin carries the remainder's sign
  const uint32_t csign = (((q + 1u) & 2u) << 30) ^ (swap ? ssp : 0u), ssign = ((q & 2u) << 30) ^ (swap ? 0u : ssp);
  ge = f2_mul(rad, swap ? sp : cp);
  go = f2_mul(rad, swap ? cp : sp);
  ge.h = __uint_as_float(__float_as_uint(ge.h) ^ csign);
  ge.l = __uint_as_float(__float_as_uint(ge.l) ^ csign);
  go.h = __uint_as_float(__float_as_uint(go.h) ^ ssign);
  go.l = __uint_as_float(__float_as_uint(go.l) ^ ssign);
}

// ------------------------------------------------------------ rounding to u_s
template <int FMT>
__device__ __forceinline__ uint32_t round_f32(float x) {
  if constexpr (FMT == FMT_F16) {
    return (uint32_t)__half_as_ushort(__float2half_rn(x));
  } else if constexpr (FMT == FMT_BF16) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
  } else {
    return (uint32_t)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
  }
}

// Single rounding of an FP64 value: round to odd into FP32 (24 bits, at least
// two more than every target), then round to nearest even into the target.
template <int FMT>
__device__ __forceinline__ uint32_t round_f64(double g) {
  float t = __double2float_rz(g);
  if ((double)t != g) t = __uint_as_float(__float_as_uint(t) | 1u);
  return round_f32<FMT>(t);
}

// The same of h + l, |l| <= an ulp of h: round to odd from the pair, then to the target.
template <int FMT>
__device__ __forceinline__ uint32_t round_f2(float h, float l) {
  uint32_t t = __float_as_uint(h);
  if (l != 0.0f) {
    if ((__float_as_uint(l) ^ t) & 0x80000000u) t -= 1u;   // toward zero (h != 0: it dominates l)
    t |= 1u;
  }
  return round_f32<FMT>(__uint_as_float(t));
}

template <int FMT>
__device__ __forceinline__ double bits_to_double(uint32_t v) {
  if constexpr (FMT == FMT_F16) {
    return (double)__half2float(__ushort_as_half((unsigned short)v));
  } else if constexpr (FMT == FMT_BF16) {
    return (double)__bfloat162float(__ushort_as_bfloat16((unsigned short)v));
  } else {
    __half_raw hr = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)v, __NV_E4M3);
    return (double)__half2float(__half(hr));
  }
}

// The FP64 definition, rounded once into u_s.
template <int FMT>
__device__ __forceinline__ void gauss_pair_slow(uint32_t a, uint32_t b, uint32_t& be, uint32_t& bo) {
  double ge, go;
  spec_gauss_pair(a, b, ge, go);
  be = round_f64<FMT>(ge);
  bo = round_f64<FMT>(go);
}

// fl_s(G) bits of a pair the estimate left undecided: double-float, then the FP64 definition.
template <int FMT>
__device__ __forceinline__ void gauss_pair_resolve(uint32_t a, uint32_t b, uint32_t& be, uint32_t& bo) {
  F2 ge, go;
  df_gauss_pair(a, b, ge, go);
  const float de = fabsf(ge.h) * kDfRel, dodd = fabsf(go.h) * kDfRel;
  be = round_f2<FMT>(ge.h, __fsub_rn(ge.l, de));
  bo = round_f2<FMT>(go.h, __fsub_rn(go.l, dodd));
  // a quarter-turn angle has an entry of exactly zero (either sign), U1 = 1 a zero radius: by definition
  const bool ok = be == round_f2<FMT>(ge.h, __fadd_rn(ge.l, de)) && bo == round_f2<FMT>(go.h, __fadd_rn(go.l, dodd)) &&
                  ge.h != 0.0f && go.h != 0.0f && a != 0xFFFFFFFFu;
  if (!ok) gauss_pair_slow<FMT>(a, b, be, bo);
}

// fl_s(G) bits of the two entries served by one (a, b) word pair.
template <int FMT>
__device__ __forceinline__ void gauss_pair_bits(uint32_t a, uint32_t b, uint32_t& be, uint32_t& bo) {
  uint32_t w;
  if (gauss_pair_est<FMT>(a, b, w)) {
    constexpr int kBits = (FMT == FMT_E4M3) ? 8 : 16;
    be = w & ((1u << kBits) - 1u);
    bo = w >> kBits;
  } else {
    gauss_pair_resolve<FMT>(a, b, be, bo);
  }
}

}  // namespace lsq
