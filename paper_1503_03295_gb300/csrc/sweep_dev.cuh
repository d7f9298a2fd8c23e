// sweep_dev.cuh -- per-site decision of step (B) of Sec. 2.1 (Metropolis update under the
// switched Hamiltonian H' of Eq. (4)), shared by the single-lattice and batched sweeps.
//
// Proposal for site i at MC step t: Philox tag PROPOSE, counter (i, t, a); attempt a uses
// words 0, 1 for Marsaglia's sphere point and word 2 of the successful attempt is the
// acceptance uniform u; 64 failed attempts keep the spin.  The move is accepted iff
// u < exp(-beta dE'), i.e. u == 0 or ln u + beta dE' < 0, with
//   beta dE' = sum_{surviving j} [beta V(S', S_j) - L(S') - beta V(S, S_j) + L(S)]
//              - beta J (S' - S) . sum_{nn j} S_j,
//   L = log(1 - exp(beta (V - Vmax)))   (so that beta Vbar = beta V - L, Eq. (3)).
// The decision is taken in float-float (in FP32 in the FP32-guarded form) with a bound on the
// rounding error of the margin; a site whose margin is inside the bound, or whose terms are out of
// range, is settled by one warp, in FP64 and then in double-double.
#pragma once

#include <cstdint>

#include "batch.h"
#include "grid_dev.cuh"
#include "sco_internal.h"

namespace sco {
namespace {

struct SiteCtx {
  int64_t i;
  int32_t xi, yi;
  double S[3], Sn[3];
  double u;
};

// The pseudointeraction terms enter as sum_j [L_o,j - L_n,j] = log(prod z_o) - log(prod z_n)
// with z = 1 - e^x = -expm1(x): one expm1 per pair energy and two logarithms per site.  The
// products are renormalised by 2^kScale (exact) so that they never underflow.  The FP64 form's
// first decision, accept_df, compares products of e^-x - 1 instead and takes no logarithm.
constexpr int kScale64 = 600;

// p by 2^600 on the exponent field when below 2^-600, counted in sc (a multiply would be issued
// on every pair as a select); false for a subnormal or zero p (the decision then goes to the
// exact path).
__device__ __forceinline__ bool renorm600(double& p, int& sc) {
  const unsigned long long b = pos_bits(p);
  if (b >= 0x1A70000000000000ull) return true;  // 2^-600
  if ((b >> 52) == 0) return false;
  p = __longlong_as_double((long long)(b + (600ull << 52)));
  ++sc;
  return true;
}

// Pair terms from the sweep table entry (Sw64): the beta-scaled field of S_j on site i,
// f = a1 S_j - (S_j . a3 d) d, gives x = S.f - bvm = beta V(S) - beta Vmax for the old and the
// new spin (7 + 2 x 3 FP64 operations); the rounding stays far inside c0.
//
// Error bound of the margin mu = ln u + beta dE' (first order, doubled):
//   per pair, |dx| <= c0 + eps_r |x|, and c0 from the table already includes eps_r 2 beta Vmax;
//   z = -expm1(x) has relative error eps_z + |dx| / z;  log of a product of n factors adds
//   n eps_r;  the logarithms eps_f |log P|;  sum (x_new - x_old) adds 2 sum c0 (the x errors)
//   and (n + 2) eps_r sum |x_new - x_old| <= (n + 2) eps_r 2 sum bvm <= (n + 2) sum c0 (c0 >=
//   2^-51 bvm by construction).  The first-order analysis needs lin = sum_j |dx_j| / z_j small:
//   each ratio is below 2^(e(c0_j) - e(z_j) + 1) with e the exponent field, so with two z per
//   pair lin <= n 2^(dmax + 2), dmax the largest exponent difference, found with integer
//   operations; it must stay below 2^-10 or the decision is left undecided.

// The FP64 form's decision (0: reject, 1: accept, 2: undecided) in float-float on the FP32 units
// (df32.cuh), kG lanes of a warp per site; valid on the first lane of each group (sub = 0).
//
// What bounds it: FP32 issue (about 250 instructions per pair) and the gathers of the neighbours'
// spins; in FP64 the same terms were bound by the 2 FP64 lanes of an SM per clock.
//
// With y = -x = beta (Vmax - V) >= 0 and z = 1 - e^-y, the acceptance u prod z_o e^(sum (x_n - x_o))
// < prod z_n is u prod E_o < prod E_n for E = e^y - 1, since z / e^x = E: no sum of energies is
// kept.  E = 2^k m with m in (0, 1.42) (df_expm1_scaled); the products of m are renormalised to
// [1, 2) at every factor and the exponents summed as integers.
//
// Error bound of u prod E_o / prod E_n (relative, first order, doubled).  Per factor: kDfExpRelErr
// (df_expm1_scaled given y), and dy / (1 - e^-y) <= 1.42 c0 / m with |dy| <= c0 = kYRelErr a1, where
// c0 / m < 2^((d >> 23) + 1 - 40) for d the largest difference of the FP32 bit images of a1 and m
// (a difference of 2^23 is a factor of two, off by at most 2^0.09); it has to stay below 2^-9, or
// the site is left undecided (y below kYMin or above kFoldMax likewise).  The products add
// 2^-43 per factor, the exchange factor its argument's error and kDfExpRelErr.
constexpr float kDfExpRelErr = 0x1p-31f;  // largest seen 2^-31.6 (y < 8192)

// Index step from site (xi, yi) to its exchange neighbour q (0 to 3: left, right, down, up); 0: none.
__device__ __forceinline__ int32_t exch_step(const DevParams& P, int32_t xi, int32_t yi, int q) {
  if (q < 2) return q == 0 ? (xi > 0 ? -1 : 0) : (xi + 1 < P.Lx ? 1 : 0);
  return q == 2 ? (yi > 0 ? -P.Lx : 0) : (yi + 1 < P.Ly ? P.Lx : 0);
}

// X 2^K against pn, both in [1, 2), from K alone: reject (0), accept (1), undecided (2), or kByMantissa
// where the mantissas are needed.  X 2^K / pn lies between 2^(K - 1) and 2^(K + 1), and its logarithm is
// off by at most `bound` (the doubled sum of the factors' relative errors, each below 2^-5).  At low
// temperatures the sum may exceed 1, but the exponents then lie far apart: with decisions up to a bound
// of 1/4 only, the FP32 form left nearly every site to FP64 (L = 64, T = 0.005 D: 25.2 ms per sweep,
// 2.6 with all of them).
constexpr int kByMantissa = 3;
__device__ __forceinline__ int decide_far(int K, float bound) {
  if (bound < 0.25f) return K >= 2 ? 0 : K <= -2 ? 1 : kByMantissa;
  const float m = bound * 1.4427f;  // in factors of two
  return (float)(K - 1) > m ? 0 : (float)(K + 1) < -m ? 1 : 2;
}

template <int kG, bool kExch>
__device__ __forceinline__ int accept_df(const DevParams& P, int32_t xi, int32_t yi,
                                         const SpinDf& S, const SpinDf& N,
                                         const PairDf* __restrict__ pdf, const SpinDf* sd,
                                         const uint32_t* __restrict__ col, uint32_t e0,
                                         uint32_t e1, uint32_t i, int sub) {
  df pn = {1.f, 0.f}, po = {1.f, 0.f};
  int K = 0, n = 0, dmax = -0x40000000;  // K: exponent of prod E_o / prod E_n beside po / pn
  bool bad = false;
  uint32_t jn = e0 + sub < e1 ? col[e0 + sub] : 0u;  // the entry one iteration ahead
  df ws = {0.f, 0.f};  // (S' - S) . (sum of the neighbours' spins), this lane's part
  if (kExch && P.J != 0.0 && sub < 4) {
    df hx = {0.f, 0.f}, hy = hx, hz = hx;
#pragma unroll
    for (int q = 0; q < 4; q += kG < 4 ? kG : 4) {
      const int32_t k = exch_step(P, xi, yi, q + sub);
      if (k == 0) continue;
      const SpinDf b = load32(sd + (int32_t)i + k);
      hx = df_add(hx, {b.hx, b.lx});
      hy = df_add(hy, {b.hy, b.ly});
      hz = df_add(hz, {b.hz, b.lz});
    }
    ws = df_mul(df_sub({N.hx, N.lx}, {S.hx, S.lx}), hx);
    ws = df_add(ws, df_mul(df_sub({N.hy, N.ly}, {S.hy, S.ly}), hy));
    ws = df_add(ws, df_mul(df_sub({N.hz, N.lz}, {S.hz, S.lz}), hz));
  }
  for (uint32_t e = e0 + sub; e < e1; e += kG) {
    const uint32_t j = jn;
    if (e + kG < e1) jn = col[e + kG];
    if (j & kExchOnly) continue;
    int32_t xj, yj;
    site_xy(j, P, xj, yj);
    const int32_t dx = xj - xi, dy = yj - yi;
    const SpinDf b = load32(sd + j);
    const PairDf t = load32(pdf + (abs(dx) + (int64_t)P.Lx * abs(dy)));
    const FieldDf g = df_field(t, dx < 0 ? -t.ax : t.ax, dy < 0 ? -t.ay : t.ay, b);
    df yn = df_pair_y(t, g, N), yo = df_pair_y(t, g, S);
    // (the sum, not the maximum, which passes over a NaN)
    int kn, ko;
    if (!(fminf(yn.h, yo.h) > kYMin && yn.h + yo.h < 8192.f)) {
      // T from D / 2048 down to 4e-6 D; the exponents of a site add up to less than 105 beta D (the sum of
      // r^-3 is 9.04, y <= 8 beta D r^-3)
      if (!(fminf(yn.h, yo.h) > kYMin && yn.h + yo.h < kFoldMax) || P.bD > 0x1p24) {
        bad = true;
        continue;
      }
      yn = df_fold(yn, kn, 128.f);
      yo = df_fold(yo, ko, 128.f);
      K += ko - kn;
    }
    const df mn = df_expm1_scaled(yn, kn), mo = df_expm1_scaled(yo, ko);
    dmax = max(dmax, __float_as_int(t.a1h) - __float_as_int(fminf(mn.h, mo.h)));
    pn = df_mul(pn, mn);
    po = df_mul(po, mo);
    int xn = kn, xo = ko;
    df_renorm(pn, xn);
    df_renorm(po, xo);
    K += xo - xn;
    ++n;
  }
  if (kG > 1) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) {
      const df qn = {__shfl_down_sync(0xffffffffu, pn.h, o, kG),
                     __shfl_down_sync(0xffffffffu, pn.l, o, kG)};
      const df qo = {__shfl_down_sync(0xffffffffu, po.h, o, kG),
                     __shfl_down_sync(0xffffffffu, po.l, o, kG)};
      pn = df_mul(pn, qn);
      po = df_mul(po, qo);
      K += __shfl_down_sync(0xffffffffu, K, o, kG);
      n += __shfl_down_sync(0xffffffffu, n, o, kG);
      dmax = max(dmax, __shfl_down_sync(0xffffffffu, dmax, o, kG));
      bad |= __shfl_down_sync(0xffffffffu, (int)bad, o, kG) != 0;
    }
    if (kExch) {  // (whole warps: the lattices of a batch differ in J)
#pragma unroll
      for (int o = kG < 4 ? kG / 2 : 2; o > 0; o >>= 1) {
        const df q = {__shfl_down_sync(0xffffffffu, ws.h, o, kG),
                      __shfl_down_sync(0xffffffffu, ws.l, o, kG)};
        ws = df_add(ws, q);
      }
    }
  }
  if (sub != 0) return 0;
  if (N.u_h == 0.f && N.u_l == 0.f) return 1;  // u = 0 accepts outright
  if (bad) return 2;
  float bound = 0x1p-30f + (float)n * (2.f * kDfExpRelErr + 0x1p-42f);
  if (n > 0) {
    const int x = (dmax >> 23) + 1 - 40;
    if (x > -9) return 2;
    bound += 2.84f * (float)n * __int_as_float((max(x, -100) + 127) << 23);
  }
  df X = df_mul({N.u_h, N.u_l}, po);
  if (kExch && P.J != 0.0) {
    // e^tex, tex = -beta J w
    df w = df_mul(ws, {-P.bJ_h, -P.bJ_l});
    w = df_fast(w.h, w.l);
    const float aj = fabsf(P.bJ_h);
    // |w error| <= 2^-40 beta J 4 (float-float sums of 12 terms below 2 each, scaled)
    int k, k0 = 0;
    if (!(fabsf(w.h) < 8192.f)) {
      if (!(fabsf(w.h) < kFoldMax)) return 2;  // (or a NaN spin)
      w = df_fold(w, k0);
    }
    const df e = w.h < 0.f ? df_exp_core<true>(w, k) : df_exp_core<false>(w, k);
    X = df_mul(X, df_add({1.f, 0.f}, e));
    K += k + k0;
    bound += 0x1p-31f + 0x1p-38f * aj;
  }
  bound *= 2.f;
  int kx = 0, kn = 0;
  df_renorm(X, kx);
  df_renorm(pn, kn);
  K += kx - kn;
  const int far = decide_far(K, bound);
  if (far != kByMantissa) return far;
  const float f = K == 0 ? 1.f : (K > 0 ? 2.f : 0.5f);
  const float D = (X.h * f - pn.h) + (X.l * f - pn.l);
  const float lim = bound * pn.h;
  if (D < -lim) return 1;
  if (D > lim) return 0;
  return 2;
}

// The FP32-guarded form's screen: the same decision in plain FP32, from the FP32 spins and constants
// (about 60 instructions per pair).  Bound as in accept_df, with kE32RelErr, c0 = kY32RelErr a1
// (c0 / m < 2^((d >> 23) + 1 - 18), below 2^-6) and 2^-23 per product; it leaves 1.5 to 2.5 sites in
// 10^4 to FP64 (T = 0.8 to 0.3 D).  N = {S', u}.
template <int kG, bool kExch>
__device__ __forceinline__ int accept_f32(const DevParams& P, int32_t xi, int32_t yi, float4 S,
                                          float4 N, const float4* __restrict__ sw,
                                          const float4* s32, const uint32_t* __restrict__ col,
                                          uint32_t e0, uint32_t e1, uint32_t i, int sub) {
  float pn = 1.f, po = 1.f;
  int K = 0, n = 0, dmax = -0x40000000;
  bool bad = false;
  uint32_t jn = e0 + sub < e1 ? col[e0 + sub] : 0u;  // the entry one iteration ahead
  float ws = 0.f;  // (S' - S) . (sum of the neighbours' spins), this lane's part
  if (kExch && P.J != 0.0 && sub < 4) {
    float hx = 0.f, hy = 0.f, hz = 0.f;
#pragma unroll
    for (int q = 0; q < 4; q += kG < 4 ? kG : 4) {
      const int32_t k = exch_step(P, xi, yi, q + sub);
      if (k == 0) continue;
      const float4 b = s32[(int32_t)i + k];
      hx += b.x;
      hy += b.y;
      hz += b.z;
    }
    ws = (N.x - S.x) * hx + (N.y - S.y) * hy + (N.z - S.z) * hz;
  }
  for (uint32_t e = e0 + sub; e < e1; e += kG) {
    const uint32_t j = jn;
    if (e + kG < e1) jn = col[e + kG];
    if (j & kExchOnly) continue;
    int32_t xj, yj;
    site_xy(j, P, xj, yj);
    const int32_t dx = xj - xi, dy = yj - yi;
    const float4 b = s32[j];
    const float4 t = __ldg(sw + (abs(dx) + (int64_t)P.Lx * abs(dy)));  // {a1, a3, bvm, 0}
    float gx, gy, gz;
    f32_field(t.x, t.y, (float)dx, (float)dy, b.x, b.y, b.z, gx, gy, gz);
    const float yn = f32_y(t.z, gx, gy, gz, N.x, N.y, N.z);
    const float yo = f32_y(t.z, gx, gy, gz, S.x, S.y, S.z);
    if (!(fminf(yn, yo) > kYMin && yn + yo < 8192.f)) {
      bad = true;
      continue;
    }
    int kn, ko;
    const float mn = f32_expm1_scaled(yn, kn), mo = f32_expm1_scaled(yo, ko);
    dmax = max(dmax, __float_as_int(t.x) - __float_as_int(fminf(mn, mo)));
    pn *= mn;
    po *= mo;
    f32_renorm(pn, kn);
    f32_renorm(po, ko);
    K += ko - kn;
    ++n;
  }
  if (kG > 1) {
#pragma unroll
    for (int o = kG / 2; o > 0; o >>= 1) {
      pn *= __shfl_down_sync(0xffffffffu, pn, o, kG);
      po *= __shfl_down_sync(0xffffffffu, po, o, kG);
      K += __shfl_down_sync(0xffffffffu, K, o, kG);
      n += __shfl_down_sync(0xffffffffu, n, o, kG);
      dmax = max(dmax, __shfl_down_sync(0xffffffffu, dmax, o, kG));
      bad |= __shfl_down_sync(0xffffffffu, (int)bad, o, kG) != 0;
    }
    if (kExch) {  // (whole warps: the lattices of a batch differ in J)
#pragma unroll
      for (int o = kG < 4 ? kG / 2 : 2; o > 0; o >>= 1) ws += __shfl_down_sync(0xffffffffu, ws, o, kG);
    }
  }
  if (sub != 0) return 0;
  if (N.w == 0.f) return 1;  // u = 0 accepts outright
  if (bad) return 2;
  float bound = 0x1p-20f + (float)n * (2.f * kE32RelErr + 0x1p-22f);
  if (n > 0) {
    const int x = (dmax >> 23) + 1 - 18;
    if (x > -6) return 2;
    bound += 2.84f * (float)n * __int_as_float((max(x, -100) + 127) << 23);
  }
  float X = N.w * po;
  if (kExch && P.J != 0.0) {
    float w = -P.bJ_f * ws;
    const float aj = fabsf(P.bJ_f);
    int k, k0 = 0;
    if (!(fabsf(w) < 8192.f)) {
      if (!(fabsf(w) < kFoldMax)) return 2;
      w = f32_fold(w, k0);
    }
    const float e = w < 0.f ? f32_exp_core<true>(w, k) : f32_exp_core<false>(w, k);
    X *= 1.f + e;
    K += k + k0;
    // |w error|: 24 terms below 8 beta J in all, each off by less than 2^-21 relative
    bound += kE32RelErr + 0x1p-17f * aj;
  }
  bound *= 2.f;
  int kx = 0, kn = 0;
  f32_renorm(X, kx);
  f32_renorm(pn, kn);
  K += kx - kn;
  const int far = decide_far(K, bound);
  if (far != kByMantissa) return far;
  const float D = X * (K == 0 ? 1.f : (K > 0 ? 2.f : 0.5f)) - pn;
  const float lim = bound * pn;
  if (D < -lim) return 1;
  if (D > lim) return 0;
  return 2;
}

// Proposal of site i at MC step t (Philox tag PROPOSE, counter (i, t, a)); false if all 64
// attempts were rejected.
// The square root and the spin are computed once, after the attempts (whose count differs
// between the lanes of a warp).
__device__ __forceinline__ bool propose(const DevParams& P, SiteCtx& c, uint64_t step) {
  double a1, a2, s;
  W4 w;
  bool ok = false;
  for (uint64_t a = 0; a < 64 && !ok; ++a) {
    w = philox((uint64_t)c.i, step, a, kTagPropose, P.key0, P.key1);
    // 0 < s < 1 from the leading 24 bits of each word in FP32 (s off by less than 2^-20) unless it
    // is within 2^-18 of either end: the lanes of a warp go through as many attempts as the
    // unluckiest needs, and each cost three FP64 instructions (305 us for 5.3 million sites)
    const float f1 = (float)((int)(w.w[0] >> 40) - (1 << 23)) * 0x1p-23f;
    const float f2 = (float)((int)(w.w[1] >> 40) - (1 << 23)) * 0x1p-23f;
    const float f = f1 * f1 + f2 * f2;
    ok = f < 1.f;
    if (fabsf(f - 0.5f) > 0.5f - 0x1p-18f && f < 1.f + 0x1p-18f)
      ok = marsaglia_point(w.w[0], w.w[1], a1, a2, s);
  }
  if (!ok) return false;
  marsaglia_point(w.w[0], w.w[1], a1, a2, s);
  const uint64_t wu = w.w[2];
  marsaglia_spin(a1, a2, s, c.Sn[0], c.Sn[1], c.Sn[2]);
  c.u = u53(wu);
  return true;
}

// Proposals are drawn for every site before the colour classes of a step run (they depend only on
// (seed, site, step)), one double4 {S'x, S'y, S'z, u} per site; u = -1 marks a site whose 64 attempts
// were all rejected (no move).  One lattice keeps them in the order of perm, so that a class reads
// its own as one stream (by site, each class touched nearly every 64-byte pair of sectors of the
// records); a batch by global site.
__device__ __forceinline__ bool take_proposal(SiteCtx& c, const double4_32a* prop) {
  const double4_32a q = *prop;
  c.Sn[0] = q.x;
  c.Sn[1] = q.y;
  c.Sn[2] = q.z;
  c.u = q.w;
  return q.w >= 0.0;
}

__device__ __forceinline__ void load_site(const DevParams& P, SiteCtx& c, uint32_t i,
                                          const double* __restrict__ s) {
  c.i = i;
  c.yi = (int32_t)site_row(i, P);
  c.xi = (int32_t)(i - (uint32_t)c.yi * (uint32_t)P.Lx);
  c.S[0] = s[i];
  c.S[1] = s[P.N + i];
  c.S[2] = s[2 * P.N + i];
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ dd warp_sum_dd(dd v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const dd w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    v = dd_add(v, w);
  }
  return v;
}

// FP64 decision (0: reject, 1: accept, 2: undecided) with the pairs of the site spread over the 32
// lanes of a warp (partial sums, products taken to logarithms per lane, then reduced).  eps_r =
// 2^-52 (unit roundoff, with margin), eps_f = kLogRelErr for the library's log_np (inputs in
// (0, 1]), eps_z = kExpm1RelErr6 for the library's expm1_np6 (two per pair, doubled: 4 eps_z).
// Compares, minima and renormalisation tests work on the bits of positive doubles.
__device__ int accept_fp64_warp(const DevParams& P, const SiteCtx& c,
                                const Sw64* __restrict__ sw,
                                const double* __restrict__ s,
                                const uint32_t* __restrict__ row_ptr,
                                const uint32_t* __restrict__ col, int lane) {
  double bdv = 0.0, pz_o = 1.0, pz_n = 1.0, c0s = 0.0;
  int sc_o = 0, sc_n = 0, n = 0, bad = 0, dmax = -2046;
  const uint32_t e1 = row_ptr[c.i + 1];
  for (uint32_t e = row_ptr[c.i] + lane; e < e1; e += 32) {
    const uint32_t cj = col[e];
    if (cj & kExchOnly) continue;
    const uint32_t j = cj;
    const uint32_t yj = site_row(j, P);
    const int32_t dx = (int32_t)(j - yj * (uint32_t)P.Lx) - c.xi;
    const int32_t dy = (int32_t)yj - c.yi;
    const Sw64& t = sw[(int64_t)(dx < 0 ? -dx : dx) + (int64_t)P.Lx * (dy < 0 ? -dy : dy)];
    const double fx = flip_if(t.ax, dx < 0), fy = flip_if(t.ay, dy < 0);
    const double ax3 = flip_if(t.a3x, dx < 0), ay3 = flip_if(t.a3y, dy < 0);
    const double bx = s[j], by = s[P.N + j], bz = s[2 * P.N + j];
    const double tp = bx * ax3 + by * ay3;
    const double gx = t.a1 * bx - tp * fx;
    const double gy = t.a1 * by - tp * fy;
    const double gz = t.a1 * bz;
    const double xn = fma(c.Sn[0], gx, fma(c.Sn[1], gy, fma(c.Sn[2], gz, -t.bvm)));
    const double xo = fma(c.S[0], gx, fma(c.S[1], gy, fma(c.S[2], gz, -t.bvm)));
    if (!neg_strict(xn) || !neg_strict(xo)) {
      bad = 1;
      continue;
    }
    const double zn = neg_expm1_np6(xn), zo = neg_expm1_np6(xo);
    pz_n *= zn;
    pz_o *= zo;
    if (!renorm600(pz_n, sc_n) || !renorm600(pz_o, sc_o)) bad = 1;
    bdv += xn - xo;
    dmax = max(dmax, exp_field(t.c0) - min(exp_field(zn), exp_field(zo)));
    c0s += t.c0;
    ++n;
  }
  // per lane: log of its products, with the renormalisation folded in
  const double lo = log_np(pz_o) - (double)(sc_o * kScale64) * P.ln2_hi;
  const double ln = log_np(pz_n) - (double)(sc_n * kScale64) * P.ln2_hi;
  const double lsum = warp_sum_d(lo - ln);
  const double labs = warp_sum_d(fabs(lo) + fabs(ln));
  bdv = warp_sum_d(bdv);
  c0s = warp_sum_d(c0s);
  dmax = __reduce_max_sync(0xffffffffu, dmax);
  n = __reduce_add_sync(0xffffffffu, n);
  bad = __reduce_or_sync(0xffffffffu, bad);
  if (bad) return 2;
  if (n > 0 && dmax + 2 + (32 - __clz(n)) > -10) return 2;
  // n 2^(dmax + 2), the power of two from its bits (dmax + 2 <= -10 here; below -1022: 0)
  const double lin = n > 0 && dmax + 2 >= -1022
                         ? (double)n * __longlong_as_double((long long)(dmax + 2 + 1023) << 52)
                         : 0.0;
  double tex = 0.0, bex = 0.0;
  if (P.J != 0.0) {
    double h0 = 0.0, h1 = 0.0, h2 = 0.0;
    const int64_t nb[4] = {c.xi > 0 ? c.i - 1 : -1, c.xi + 1 < P.Lx ? c.i + 1 : -1,
                           c.yi > 0 ? c.i - P.Lx : -1, c.yi + 1 < P.Ly ? c.i + P.Lx : -1};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (nb[q] < 0) continue;
      h0 += s[nb[q]];
      h1 += s[P.N + nb[q]];
      h2 += s[2 * P.N + nb[q]];
    }
    const double dot = (c.Sn[0] - c.S[0]) * h0 + (c.Sn[1] - c.S[1]) * h1 + (c.Sn[2] - c.S[2]) * h2;
    tex = -(P.beta * P.J) * dot;
    bex = 0x1p-44 * fabs(P.beta * P.J);
  }
  const double lu = log_np(c.u);
  const double mu = lu + ((bdv + tex) + lsum);
  const double B = 2.0 * ((double)(n + 4) * c0s + 2.0 * lin + n * (4.0 * kExpm1RelErr6 + 0x1p-51) +
                          kLogRelErr * (labs + fabs(lu)) + 0x1p-49 * labs + bex +
                          0x1p-51 * (fabs(tex) + fabs(bdv) + fabs(mu)));
  if (mu < -B) return 1;
  if (mu > B) return 0;
  return 2;
}

// The same comparison in double-double, pairs spread over the lanes.
__device__ bool accept_dd_warp(const DevParams& P, const SiteCtx& c,
                               const double* __restrict__ s,
                               const uint32_t* __restrict__ row_ptr,
                               const uint32_t* __restrict__ col, int lane) {
  const dd ln2 = {P.ln2_hi, P.ln2_lo};
  dd sum = dd_from(0.0);
  int inf = 0;
  const uint32_t e1 = row_ptr[c.i + 1];
  for (uint32_t e = row_ptr[c.i] + lane; e < e1; e += 32) {
    const uint32_t cj = col[e];
    if (cj & kExchOnly) continue;
    const uint32_t j = cj;
    const uint32_t yj = site_row(j, P);
    const int32_t dx = (int32_t)(j - yj * (uint32_t)P.Lx) - c.xi;
    const int32_t dy = (int32_t)yj - c.yi;
    const int64_t r2 = (int64_t)dx * dx + (int64_t)dy * dy;
    const double cc = coupling_c(r2);
    const dd Vm = dd_vmax(P.D, hazard_A(r2));
    const double Sj[3] = {s[j], s[P.N + j], s[2 * P.N + j]};
    const dd Vn = dd_pair_V(P.D, cc, (double)r2, c.Sn, Sj, (double)dx, (double)dy);
    const dd Vo = dd_pair_V(P.D, cc, (double)r2, c.S, Sj, (double)dx, (double)dy);
    const dd xn = dd_mul_d(dd_sub(Vn, Vm), P.beta);
    const dd xo = dd_mul_d(dd_sub(Vo, Vm), P.beta);
    if (!(xn.hi < 0.0)) {  // Vbar(S') = +inf
      inf = 1;
      continue;
    }
    sum = dd_add(sum, dd_mul_d(dd_sub(Vn, Vo), P.beta));
    sum = dd_sub(sum, dd_log1mexp(xn, ln2));
    sum = dd_add(sum, dd_log1mexp(xo, ln2));
  }
  sum = warp_sum_dd(sum);
  if (__reduce_or_sync(0xffffffffu, inf)) return false;
  if (P.J != 0.0) {
    dd h[3] = {dd_from(0.0), dd_from(0.0), dd_from(0.0)};
    const int64_t nb[4] = {c.xi > 0 ? c.i - 1 : -1, c.xi + 1 < P.Lx ? c.i + 1 : -1,
                           c.yi > 0 ? c.i - P.Lx : -1, c.yi + 1 < P.Ly ? c.i + P.Lx : -1};
    for (int q = 0; q < 4; ++q) {
      if (nb[q] < 0) continue;
      for (int a = 0; a < 3; ++a) h[a] = dd_add(h[a], dd_from(s[a * P.N + nb[q]]));
    }
    dd dot = dd_from(0.0);
    for (int a = 0; a < 3; ++a) dot = dd_add(dot, dd_mul(two_sum(c.Sn[a], -c.S[a]), h[a]));
    sum = dd_sub(sum, dd_mul(dot, two_prod(P.beta, P.J)));
  }
  const dd lu = dd_log(dd_from(c.u), ln2);
  return dd_lt(dd_add(lu, sum), dd_from(0.0));
}


// ---- the sweep of a whole MC step, one lattice or a batch ----------------------------------
// One persistent cooperative kernel walks the colours in ascending order, one grid barrier apart
// (a launch per colour took 6 to 7 us for a small class, most of it launch and drain).  The trailing
// colours that hold at most kTailSites sites each are left to block 0, one __syncthreads apart.
// Sweep phase per step, with a launch per colour, FP64 terms on the FP64 units and the old spins'
// terms kept by the switch, and now: L = 2304 FP64 6.98 -> 1.92 ms, FP32-guarded 2.42 -> 1.31, L = 1152
// with exchange, FP64 1.02 -> 0.35, L = 256 FP64 0.83 -> 0.12.
constexpr int kSweepThreads = 512;
constexpr uint32_t kTailSites = 64;

struct SweepView {
  int R;                       // lattices
  const uint32_t* site_start;  // R + 1 (batch)
  const RepDesc* desc;         // R (batch)
  DevParams P;                 // one lattice: its parameters and tables
  const PairDf* pdf;
  const float4* sw32;
  const Sw64* sw;
  double* s;
  float4* s32;
  SpinDf* sd;
  const uint32_t* row_ptr;
  const uint32_t* col;
  const uint32_t* perm;        // sites by colour, global indices
  const uint32_t* off;         // class starts, g + 1
  const double4_32a* prop;     // proposals {S', u}, FP64 (see take_proposal)
  const SpinDf* propd;         // and in float-float (FP64 form)
  const float4* prop32;        // or FP32 (FP32-guarded form)
  uint8_t* acc;
  DevCounters* cnt;            // R
  uint32_t g;                  // colours
  const unsigned* gmax;        // or on the device (batch)
  unsigned* bar;
  int* status;
  const int* halt;             // optional: nonzero on entry -> return at once
  unsigned long long ns_limit;
};

// One site's decision in FP64 then double-double by a whole warp, for the sites that the first
// decision leaves open: a function of its own, so that its registers stay out of the sweep.
__device__ __noinline__ bool settle_site(const DevParams& P, uint32_t i,
                                         const Sw64* __restrict__ sw, const double* s,
                                         const uint32_t* __restrict__ row_ptr,
                                         const uint32_t* __restrict__ col,
                                         const double4_32a* prop, int lane, unsigned& ndd) {
  SiteCtx c;
  load_site(P, c, i, s);
  take_proposal(c, prop);
  int d = accept_fp64_warp(P, c, sw, s, row_ptr, col, lane);
  if (d == 2) {
    ++ndd;
    d = accept_dd_warp(P, c, s, row_ptr, col, lane) ? 1 : 0;
  }
  return d == 1;
}

// The n sites perm[b ..], kG lanes per site, warps w, w + nw, ...; undecided sites are settled at once
// by their warp.  sbase: site bases in shared memory (batch); sg: counters of screened-out and
// double-double decisions (batch: per lattice, one lattice: none) beside n32 and ndd.
template <int kPrec, bool kBatch, bool kExch, int kG>
__device__ __forceinline__ void sweep_class(const SweepView& V, const uint32_t* sbase, uint32_t* sg,
                                            uint32_t b, uint32_t n, uint32_t w, uint32_t nw,
                                            unsigned& n32, unsigned& ndd) {
  constexpr uint32_t kSites = 32 / kG;
  const int lane = threadIdx.x & 31, sub = lane % kG;
  for (uint32_t q = w * kSites; q < n; q += nw * kSites) {
    const uint32_t idx = q + lane / kG;
    uint32_t gs = 0, base = 0, e0 = 0, e1 = 0;
    int r = 0;
    if (idx < n) {
      gs = V.perm[b + idx];
      if (kBatch) {
        r = find_le(sbase, V.R, gs);
        base = sbase[r];
      }
    }
    const RepDesc* dr = kBatch ? V.desc + r : nullptr;
    const DevParams& P = kBatch ? dr->P : V.P;
    const uint32_t i = gs - base;
    int32_t xi, yi;
    site_xy(i, P, xi, yi);
    SpinDf Nd;
    float4 N4;
    bool move;
    int d;
    if (kPrec == 0) {
      SpinDf S;
      Nd.u_h = -1.f;
      if (idx < n) {
        Nd = load32(V.propd + (kBatch ? gs : b + idx));
        e0 = V.row_ptr[gs];
        e1 = V.row_ptr[gs + 1];
        S = load32(V.sd + gs);
      }
      move = Nd.u_h >= 0.f;
      if (!move) e1 = e0;
      d = accept_df<kG, kExch>(P, xi, yi, S, Nd, kBatch ? dr->pdf : V.pdf, V.sd + base, V.col, e0, e1, i,
                               sub);
    } else {
      float4 S;
      N4.w = -1.f;
      if (idx < n) {
        N4 = V.prop32[kBatch ? gs : b + idx];
        e0 = V.row_ptr[gs];
        e1 = V.row_ptr[gs + 1];
        S = V.s32[gs];
      }
      move = N4.w >= 0.f;
      if (!move) e1 = e0;
      d = accept_f32<kG, kExch>(P, xi, yi, S, N4, kBatch ? dr->sw32 : V.sw32, V.s32 + base, V.col, e0,
                                e1, i, sub);
    }
    const bool mine = sub == 0 && idx < n;
    if (!mine || !move) d = 0;
    for (unsigned open = __ballot_sync(0xffffffffu, d == 2); open != 0; open &= open - 1) {
      const int src = __ffs(open) - 1;
      const uint32_t gi = __shfl_sync(0xffffffffu, gs, src);
      uint32_t bi = 0;
      int ri = 0;
      if (kBatch) {
        ri = find_le(sbase, V.R, gi);
        bi = sbase[ri];
      }
      const RepDesc* di = kBatch ? V.desc + ri : nullptr;
      unsigned dd = 0;
      const bool ok = settle_site(kBatch ? di->P : V.P, gi - bi, kBatch ? di->sw64 : V.sw,
                                  V.s + 3 * (size_t)bi, V.row_ptr + bi, V.col,
                                  V.prop + (kBatch ? gi : b + q + src / kG), lane, dd);
      if (lane == src) {
        d = ok ? 1 : 0;
        if (kBatch) {
          if (kPrec == 1) atomicAdd(&sg[2 * ri], 1u);
          if (dd) atomicAdd(&sg[2 * ri + 1], dd);
        } else {
          n32 += kPrec == 1 ? 1u : 0u;
          ndd += dd;
        }
      }
    }
    if (mine) {
      if (d == 1) {
        const double4_32a v = V.prop[kBatch ? gs : b + idx];
        double* s = V.s + 3 * (size_t)base;
        s[i] = v.x;
        s[P.N + i] = v.y;
        s[2 * P.N + i] = v.z;
        if (kPrec == 0) V.sd[gs] = Nd;
        else V.s32[gs] = make_float4(N4.x, N4.y, N4.z, 0.f);
      }
      V.acc[gs] = d == 1 ? 1 : 0;
    }
  }
}

// Lanes per site: 2 while the class gives every second lane a site (one lane per site took 2.37 ms
// per step at L = 2304 in the FP64 form, two 2.20, four 2.28), 8 and 32 below, where the class would
// leave lanes idle and a row's serial chain sets the time.
__device__ __forceinline__ uint32_t sweep_lanes(uint32_t n, uint32_t nw) {
  return n >= nw * 16 ? 2 : n >= nw ? 8 : 32;
}
template <int kPrec, bool kBatch, bool kExch>
__device__ __forceinline__ void sweep_tiers(const SweepView& V, const uint32_t* sbase, uint32_t* sg,
                                            uint32_t b, uint32_t n, uint32_t w, uint32_t nw,
                                            unsigned& n32, unsigned& ndd) {
  const uint32_t k = sweep_lanes(n, nw);
  if (k == 2) sweep_class<kPrec, kBatch, kExch, 2>(V, sbase, sg, b, n, w, nw, n32, ndd);
  else if (k == 8) sweep_class<kPrec, kBatch, kExch, 8>(V, sbase, sg, b, n, w, nw, n32, ndd);
  else sweep_class<kPrec, kBatch, kExch, 32>(V, sbase, sg, b, n, w, nw, n32, ndd);
}

inline size_t sweep_smem(int R) { return (size_t)(3 * R + 1) * sizeof(uint32_t); }

template <int kPrec, bool kBatch, bool kExch, int kBlocks>
__global__ void __launch_bounds__(kSweepThreads, kBlocks) k_sweep(const __grid_constant__ SweepView V) {
  __shared__ int s_halt;
  __shared__ unsigned s_tail;
  if (threadIdx.x == 0) {
    // an error before this step (a colouring whose wait ran out): the classes may not be there
    s_halt = (V.halt && ld_status(V.halt)) || ld_status(V.status);
    s_tail = 0;
  }
  __syncthreads();
  if (s_halt) return;
  extern __shared__ uint32_t wsm[];
  uint32_t* sbase = wsm;         // R + 1 (batch)
  uint32_t* sg = wsm + V.R + 1;  // 2 R (batch)
  if (kBatch) {
    for (int r = threadIdx.x; r <= V.R; r += blockDim.x) sbase[r] = V.site_start[r];
    for (int r = threadIdx.x; r < 2 * V.R; r += blockDim.x) sg[r] = 0;
  }
  const uint32_t g = V.gmax ? *V.gmax : V.g;
  // class starts in shared memory: the barrier drops what L1 holds
  constexpr uint32_t kOffs = 256;
  __shared__ uint32_t soff[kOffs + 1];
  for (uint32_t c = threadIdx.x; c <= min(g, kOffs); c += blockDim.x) soff[c] = V.off[c];
  for (uint32_t c = threadIdx.x; c < g; c += blockDim.x)
    if (V.off[c + 1] - V.off[c] > kTailSites) atomicMax(&s_tail, c + 1);
  __syncthreads();
  const uint32_t tail = s_tail;  // colours from here on are small
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  unsigned n32 = 0, ndd = 0;
  bool ok = true;
  uint32_t b = soff[0];
  for (uint32_t c = 0; c < tail && ok; ++c) {
    const uint32_t e = c + 1 <= kOffs ? soff[c + 1] : V.off[c + 1];
    if (e > b) {
      sweep_tiers<kPrec, kBatch, kExch>(V, sbase, sg, b, e - b, w, (gridDim.x * blockDim.x) >> 5, n32,
                                        ndd);
      if (gridDim.x > 1) ok = grid_sync(V.bar, V.status, V.ns_limit);
      else __syncthreads();
    }
    b = e;
  }
  if (blockIdx.x == 0 && ok) {
    for (uint32_t c = tail; c < g; ++c) {
      const uint32_t e = c + 1 <= kOffs ? soff[c + 1] : V.off[c + 1];
      if (e > b) {
        sweep_tiers<kPrec, kBatch, kExch>(V, sbase, sg, b, e - b, w, kSweepThreads / 32, n32, ndd);
        __syncthreads();
      }
      b = e;
    }
  }
  if (kBatch) {
    __syncthreads();
    for (int r = threadIdx.x; r < V.R; r += blockDim.x) {
      if (sg[2 * r]) atomicAdd(&V.cnt[r].guard_fp32, (unsigned long long)sg[2 * r]);
      if (sg[2 * r + 1]) atomicAdd(&V.cnt[r].guard_fp64, (unsigned long long)sg[2 * r + 1]);
    }
  } else {
    if (n32) atomicAdd(&V.cnt->guard_fp32, (unsigned long long)n32);
    if (ndd) atomicAdd(&V.cnt->guard_fp64, (unsigned long long)ndd);
  }
}

// Resident blocks per SM for `sites` sites: two (64 registers; three at 42 in FP32: 1.59 ms per step
// at L = 2304 against 1.66) on a large lattice or batch; below kSweepWide sites per SM one, at 128
// registers and without spills (L = 256: 0.130 ms per step against 0.163, L = 1024: 0.642 against
// 0.594; 10 lattices of L = 128, FP32, with the
// proposals: 95 us against 111), a block per kSweepSites sites, so that its
// barriers have few blocks to wait for, and up to kSweepOne sites a single one.
constexpr int64_t kSweepWide = 2048, kSweepSites = 256, kSweepOne = 2048;
inline int sweep_blocks(int64_t sites, int precision) {
  return sites < kSweepWide * num_sms() ? 1 : precision == 1 ? 3 : 2;
}
template <bool kBatch, bool kExch>
const void* sweep_kernel(int precision, int per) {
  return precision == 1 ? (per > 1 ? (const void*)k_sweep<1, kBatch, kExch, 3>
                                   : (const void*)k_sweep<1, kBatch, kExch, 1>)
                        : (per > 1 ? (const void*)k_sweep<0, kBatch, kExch, 2>
                                   : (const void*)k_sweep<0, kBatch, kExch, 1>);
}

// A site's proposal for MC step `step` in the forms the sweep reads (see take_proposal).
__device__ __forceinline__ void write_proposal(const DevParams& P, uint64_t step, uint32_t i,
                                               double4_32a* prop, SpinDf* propd, float4* prop32) {
  SiteCtx c;
  c.i = i;
  const bool ok = propose(P, c, step);
  *prop = ok ? make_double4_32a(c.Sn[0], c.Sn[1], c.Sn[2], c.u)
             : make_double4_32a(0.0, 0.0, 1.0, -1.0);
  if (propd) {
    SpinDf d = proposal_df(c.Sn[0], c.Sn[1], c.Sn[2], c.u);
    if (!ok) d.u_h = -1.f;
    *propd = d;
  }
  if (prop32)
    *prop32 = make_float4((float)c.Sn[0], (float)c.Sn[1], (float)c.Sn[2], ok ? (float)c.u : -1.f);
}

}  // namespace
}  // namespace sco
