// df32.cuh -- float-float arithmetic (a value as the unevaluated sum of two FP32 numbers, about
// 48 bits) for the pair terms of the FP64 decisions.
//
// Why: an sm_103a SM issues 128 FP32 lane-operations per clock but only 2 in FP64, so an FP64
// instruction costs as much as 64 FP32 ones.  A float-float product is 4 FP32 instructions and a
// sum 8, so a pair term of the sweep (28 FP64 instructions, 1792 FP32 slots) takes about 250.
// The error-free sums and products are Knuth's and Dekker's (Dekker 1971; Ogita, Rump and Oishi
// 2005).  A sum or product here leaves its low part unnormalised and drops products of two low
// parts; with |l| <= 2^-20 |h| (or the scale of a cancelling sum) that is below 2^-40 of the scale.
#pragma once

#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace sco {

struct df {
  float h, l;
};

// The spin of a site in float-float, one 32-byte sector: components x, y, z as h + l within 2^-47.
struct __align__(32) SpinDf {
  float hx, hy, hz, u_h;  // u_h, u_l: the acceptance uniform where the record holds a proposal
  float lx, ly, lz, u_l;
};

// Pair constants at (|dx|, |dy|), one 32-byte sector: a1 = beta D c r^2, a3 = 3 beta D c and
// bvm = beta Vmax in float-float (the splits of the FP64 constants of Sw64), |dx| and |dy|.
struct __align__(32) PairDf {
  float a1h, a1l, a3h, a3l, bvmh, bvml, ax, ay;
};

__host__ __device__ __forceinline__ float df_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}
__host__ __device__ __forceinline__ float df_fmul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  volatile float p = a * b;  // not contracted into an FMA
  return p;
#endif
}
__host__ __device__ __forceinline__ uint32_t df_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float df_from_bits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

__host__ __device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__host__ __device__ __forceinline__ df df_fast(float a, float b) {  // |a| >= |b| or a = 0
  const float s = a + b;
  return {s, b - (s - a)};
}
__host__ __device__ __forceinline__ df df_mul(df a, df b) {
  const float p = df_fmul(a.h, b.h);
  return {p, df_fma(a.l, b.h, df_fma(a.h, b.l, df_fma(a.h, b.h, -p)))};
}
__host__ __device__ __forceinline__ df df_mul_f(df a, float f) {
  const float p = df_fmul(a.h, f);
  return {p, df_fma(a.l, f, df_fma(a.h, f, -p))};
}
__host__ __device__ __forceinline__ df df_add(df a, df b) {
  const df s = df_two_sum(a.h, b.h);
  return {s.h, s.l + (a.l + b.l)};
}
__host__ __device__ __forceinline__ df df_sub(df a, df b) {
  const df s = df_two_sum(a.h, -b.h);
  return {s.h, s.l + (a.l - b.l)};
}

// x as h + l from its bits: h the leading 24 bits (truncated), l the other 29 rounded to 24, so
// |x - h - l| <= 2^-47 |x|; below 2^-60 (and for x = 0) both are 0.  Integer operations and one
// conversion: a pair of FP64 conversions would cost more on the FP64 pipe.  |x| < 2^60.
__host__ __device__ __forceinline__ df df_split(double x) {
#ifdef __CUDA_ARCH__
  const uint64_t b = (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
#endif
  const int e = (int)((b >> 52) & 0x7FFu);
  if (e < 1023 - 60) return {0.f, 0.f};
  const uint32_t sg = (uint32_t)(b >> 32) & 0x80000000u;
  const float h =
      df_from_bits(sg | ((uint32_t)(e - 1023 + 127) << 23) | ((uint32_t)(b >> 29) & 0x7FFFFFu));
  const float l = (float)((uint32_t)b & 0x1FFFFFFFu) *
                  df_from_bits(sg | ((uint32_t)(e - 1075 + 127) << 23));
  return {h, l};
}
// The same for a table constant of any size (set-up only): both parts rounded.
__host__ __device__ __forceinline__ df df_split_const(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

// e^y = 2^k (1 + e0) for |y| < 8192 (y normalised; kNeg: y <= 0, else y >= 0): k is the integer
// nearest to y / ln 2 (less 0.1 for y >= 0, so that k = 0, beside which e^y - 1 cancels most,
// reaches to 0.416); r = y - k ln 2 in float-float with ln 2 = L1 + L2 + L3 (L1 and L2 of 10 bits:
// their products with |k| < 2^14 are exact), e0 = e^r - 1 = r + r^2 (1/2 + r (1/6 + r w(r))).  r w
// is below 0.02, so FP32 is enough for w; the steps above it are float-float.  w is the degree-4
// interpolant of (e^r - 1 - r - r^2/2 - r^3/6) / r^4 at the Chebyshev points of [-0.282, 0.422]
// (kNeg: [-0.352, 0.352]).
constexpr float kDfLog2e = 1.44269504088896341f;
constexpr float kDfL1 = 0x1.628p-1f;   // ln 2 to 10 bits
constexpr float kDfL2 = 0x1.908p-11f;  // the next 10
constexpr float kDfL3 = 0x1.fdf474p-22f;   // the rest
constexpr float kDfSixthL = -0x1.555556p-28f;  // 1/6 - fl(1/6)

template <bool kNeg>
__host__ __device__ __forceinline__ df df_exp_core(df y, int& k) {
  const float t =  // 1.5 2^23 + k
      kNeg ? df_fma(y.h, kDfLog2e, 12582912.f) : df_fma(y.h, kDfLog2e, -0.1f) + 12582912.f;
  const float kf = t - 12582912.f;
  k = (int)df_bits(t) - 0x4B400000;
  const float r0 = df_fma(-kf, kDfL1, y.h);
  const df s = df_two_sum(r0, -df_fmul(kf, kDfL2));
  const df r = df_fast(s.h, s.l + df_fma(-kf, kDfL3, y.l));
  constexpr float w0 = kNeg ? 0.0416666666667f : 0.0416666674795f,
                  w1 = kNeg ? 0.00833332017177f : 0.00833332586646f,
                  w2 = kNeg ? 0.00138888758013f : 0.00138880498834f,
                  w3 = kNeg ? 0.00019883945f : 0.000198706958715f,
                  w4 = kNeg ? 2.4843860e-5f : 2.58313215769e-5f;
  const float w = df_fma(df_fma(df_fma(df_fma(w4, r.h, w3), r.h, w2), r.h, w1), r.h, w0);
  const float sixth = 0x1.555556p-3f;
  df v;  // 1/6 + r w with the product's rounding kept
  v.h = df_fma(r.h, w, sixth);
  v.l = df_fma(r.h, w, sixth - v.h) + kDfSixthL;
  const df u = df_mul(r, v);
  df q;
  q.h = 0.5f + u.h;
  q.l = ((0.5f - q.h) + u.h) + u.l;
  const df r2 = {df_fmul(r.h, r.h), 0.f};
  const df r2f = {r2.h, df_fma(r.h + r.h, r.l, df_fma(r.h, r.h, -r2.h))};
  const df p = df_mul(r2f, q);
  const float eh = r.h + p.h;
  return {eh, (p.h - (eh - r.h)) + (r.l + p.l)};
}

// y by a multiple of 8192 ln 2 into the range of df_exp_core (a little across 0 at most), the multiple's
// power of two in k, for |y| < kFoldMax: q below 2^8 and L1, L2 of 10 bits, so both products and the first
// difference are exact; the rest is off by less than 2^-43 |y|.  keep: what at least remains of a
// larger y (with 128, df_expm1_scaled's 2^-k stays 0).
constexpr float kFoldMax = 0x1p20f, kDfFoldInv = 1.f / 5678.26170f;
__host__ __device__ __forceinline__ df df_fold(df y, int& k, float keep = 0.f) {
  const int q = (int)((y.h - keep) * kDfFoldInv);
  const float kf = (float)q * 8192.f;
  k = q * 8192;
  const df s = df_two_sum(df_fma(-kf, kDfL1, y.h), -df_fmul(kf, kDfL2));
  return df_fast(s.h, s.l + df_fma(-kf, kDfL3, y.l));
}
// the same in plain FP32, off by less than 2^-23 |y|
__host__ __device__ __forceinline__ float f32_fold(float y, int& k) {
  const int q = (int)(y * kDfFoldInv);
  const float kf = (float)q * 8192.f;
  k = q * 8192;
  return df_fma(-kf, kDfL2 + kDfL3, df_fma(-kf, kDfL1, y));
}

// 2^-k for k >= 0 (0 above 126)
__host__ __device__ __forceinline__ float df_pow2_neg(int k) {
  return k > 126 ? 0.f : df_from_bits((uint32_t)(127 - k) << 23);
}

// (e^y - 1) 2^-k = e0 + (1 - 2^-k) for y >= 0 (k >= 0): in (0, 1.42), with the exponent k apart
__host__ __device__ __forceinline__ df df_expm1_scaled(df y, int& k) {
  const df e = df_exp_core<false>(y, k);
  const float t = df_pow2_neg(k);
  const float ch = 1.f - t, cl = (1.f - ch) - t;
  const float mh = ch + e.h;  // |ch| >= |e.h| for k >= 1, ch = 0 for k = 0
  return {mh, (e.h - (mh - ch)) + (cl + e.l)};
}

// 1 - e^-y for y >= 0
__host__ __device__ __forceinline__ df df_one_minus_exp_neg(df y) {
  int k;
  const df e = df_exp_core<true>({-y.h, -y.l}, k);
  const float s = df_pow2_neg(-k);  // 2^k, k <= 0
  const float ch = 1.f - s, cl = (1.f - ch) - s;
  const float eh = s * e.h, el = s * e.l;  // exact scalings (or both negligible)
  const float mh = ch - eh;
  return {mh, ((ch - mh) - eh) + (cl - el)};
}

// The record of a proposal: a spin of length 1 and its acceptance uniform.
__host__ __device__ __forceinline__ SpinDf proposal_df(double x, double y, double z, double u) {
  const df a = df_split(x), b = df_split(y), c = df_split(z), w = df_split(u);
  return {a.h, b.h, c.h, w.h, a.l, b.l, c.l, w.l};
}
// The record of a spin, which may be one that a caller set.  The error bounds below are for |S| <= 1;
// up to kUnitMax per component (|S|^2 <= 3.01) the errors of the pair terms grow threefold, within the
// factors that the decisions hold in hand.  Beyond (infinite or not a number among them) the components
// are NaN, and every decision that reads them is left to FP64 and double-double.
constexpr double kUnitMax = 1.0 + 0x1p-10;
__host__ __device__ __forceinline__ bool spin_in_bounds(double x, double y, double z) {
  return x >= -kUnitMax && x <= kUnitMax && y >= -kUnitMax && y <= kUnitMax && z >= -kUnitMax &&
         z <= kUnitMax;
}
__host__ __device__ __forceinline__ SpinDf spin_df(double x, double y, double z, double u) {
  if (spin_in_bounds(x, y, z)) return proposal_df(x, y, z, u);
  const float nan = df_from_bits(0x7FC00000u);
  return {nan, nan, nan, 0.f, nan, nan, nan, 0.f};
}

// The beta-scaled field of spin b (at displacement (sx |dx|, sy |dy|), t its pair constants) on the
// other site: g = a1 S_b - a3 (S_b . d) d.  Then y = beta (Vmax - V) = bvm - S . g.
struct FieldDf {
  df x, y, z;
};
__host__ __device__ __forceinline__ FieldDf df_field(const PairDf& t, float fx, float fy,
                                                     const SpinDf& b) {
  const df a1 = {t.a1h, t.a1l}, a3 = {t.a3h, t.a3l};
  const df bx = {b.hx, b.lx}, by = {b.hy, b.ly}, bz = {b.hz, b.lz};
  const df q = df_add(df_mul_f(bx, fx), df_mul_f(by, fy));
  const df w = df_mul(a3, q);
  return {df_sub(df_mul(a1, bx), df_mul_f(w, fx)), df_sub(df_mul(a1, by), df_mul_f(w, fy)),
          df_mul(a1, bz)};
}

// y = bvm - S . g, normalised.  |error| <= kYRelErr a1 against the exact beta (Vmax - V) of the
// FP64 spins (48-bit inputs, unnormalised sums): the roundings' bounds added up along the computation
// reach 2^-40.1 a1 over 3 million pairs, the errors 2^-41.9 a1.
constexpr float kYRelErr = 0x1p-40f;
// and for y above kYMin: a1 >= y / 12 then (|S|^2 <= 3.01), so that a3 = 3 a1 / r^2, r < 2^15.6, is above
// 2^-94 and its low part, 2^-24 of it, well above the smallest FP32 number, 2^-149 (below, far pairs'
// errors reach past kYRelErr a1).
constexpr float kYMin = 0x1p-60f;
__host__ __device__ __forceinline__ df df_pair_y(const PairDf& t, const FieldDf& g,
                                                 const SpinDf& s) {
  df y = df_sub({t.bvmh, t.bvml}, df_mul(g.x, {s.hx, s.lx}));
  y = df_sub(y, df_mul(g.y, {s.hy, s.ly}));
  y = df_sub(y, df_mul(g.z, {s.hz, s.lz}));
  return df_fast(y.h, y.l);
}

// ---- the same pair term in plain FP32 (FP32-guarded form) --------------------------------
// g = a1 S_b - a3 (S_b . d) d from FP32 spins and constants, y = bvm - S . g.  |error| <= kY32RelErr
// a1 against the exact value of the FP64 spins: the spins' rounding (2^-25 per component) contributes
// 12 2^-25 a1, the constants' and the 13 operations' below 40 2^-24 a1 (every intermediate is at most
// 6 a1); added up along the computation they reach 2^-18.8 a1, the errors 2^-19.8 a1.
constexpr float kY32RelErr = 0x1p-18f;
__host__ __device__ __forceinline__ void f32_field(float a1, float a3, float fx, float fy, float bx,
                                                   float by, float bz, float& gx, float& gy,
                                                   float& gz) {
  const float w = a3 * df_fma(bx, fx, df_fmul(by, fy));
  gx = df_fma(a1, bx, -df_fmul(w, fx));
  gy = df_fma(a1, by, -df_fmul(w, fy));
  gz = a1 * bz;
}
__host__ __device__ __forceinline__ float f32_y(float bvm, float gx, float gy, float gz, float sx,
                                                float sy, float sz) {
  return df_fma(-sx, gx, df_fma(-sy, gy, df_fma(-sz, gz, bvm)));
}
// e^y = 2^k (1 + e0) for |y| < 8192, as df_exp_core (kNeg likewise); e0 by its series to r^8.
template <bool kNeg>
__host__ __device__ __forceinline__ float f32_exp_core(float y, int& k) {
  const float t =
      kNeg ? df_fma(y, kDfLog2e, 12582912.f) : df_fma(y, kDfLog2e, -0.1f) + 12582912.f;
  const float kf = t - 12582912.f;
  k = (int)df_bits(t) - 0x4B400000;
  const float r = df_fma(-kf, kDfL2 + kDfL3, df_fma(-kf, kDfL1, y));
  float w = df_fma(1.f / 40320.f, r, 1.f / 5040.f);
  w = df_fma(w, r, 1.f / 720.f);
  w = df_fma(w, r, 1.f / 120.f);
  w = df_fma(w, r, 1.f / 24.f);
  w = df_fma(w, r, 1.f / 6.f);
  w = df_fma(w, r, 0.5f);
  return df_fma(df_fmul(r, r), w, r);
}
// (e^y - 1) 2^-k for y >= 0, in (0, 1.42); relative error (given y < 8192) below kE32RelErr, the
// largest seen 2^-21.8 (y < 60: 2^-23.2)
constexpr float kE32RelErr = 0x1p-20f;
__host__ __device__ __forceinline__ float f32_expm1_scaled(float y, int& k) {
  const float e = f32_exp_core<false>(y, k);
  return (1.f - df_pow2_neg(k)) + e;
}

// p by a power of two into [1, 2) (p.h > 0 normal), the exponent added to e
__device__ __forceinline__ void df_renorm(df& p, int& e) {
  const int b = __float_as_int(p.h), x = (b >> 23) - 127;
  p.h = __int_as_float(b - (x << 23));
  p.l *= __int_as_float((127 - x) << 23);
  e += x;
}

__device__ __forceinline__ void f32_renorm(float& p, int& e) {
  const int b = __float_as_int(p), x = (b >> 23) - 127;
  p = __int_as_float(b - (x << 23));
  e += x;
}

// One 32-byte load (ld.global.v4.f64) of a record.
template <class T>
__device__ __forceinline__ T load32(const T* p) {
  static_assert(sizeof(T) == 32, "one sector");
  const double4_32a v = *reinterpret_cast<const double4_32a*>(p);
  T t;
  memcpy(&t, &v, 32);
  return t;
}

}  // namespace sco
