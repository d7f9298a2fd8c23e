// switch_dev.cuh -- per-site body of step (A) of Sec. 2.1 (potential switching), shared by
// the single-lattice and the batched switch kernels.
//
// Every pair {i, i+d} survives (V -> Vbar) with probability 1 - P_ij, P_ij of Eq. (2),
// independently.  Site i visits its half-plane list by bound thinning: element m becomes a
// candidate with probability q_m = 1 - exp(-2 beta Vmax_m) (a Poisson process of rate
// beta D A_m 2^-58 per element, walked over the prefix W), and a candidate survives with
// probability (1 - P_ij) / q_m.  The draws come from Philox tag SWITCH, counter
// (i, epoch, n/2), draw n using words 2(n%2) (exponential) and 2(n%2)+1 (survival).
//
// Every decision is an exact comparison of reals built from FP64 inputs.  It is taken in
// float-float (after FP32 in the FP32-guarded form) together with a bound on the rounding error; a
// margin inside the bound sends the decision to double-double arithmetic.
#pragma once

#include <cstdint>

#include "sco_internal.h"

namespace sco {
namespace {

constexpr int kStatusCapacity = 7;

__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// The sorted half-plane list as a walk reads it: displacements d, the hazard prefix W and the decay
// bits E of Table::Ebits, the first nnear displacements and decay bits in shared memory, and the
// guides into E (see Search).
struct NearTable {
  const uint64_t* sE;
  const uint32_t* sD;
  const uint16_t* sG;  // near guide: kNearGuide + 1 entries
  const uint64_t* W;
  const uint64_t* E;
  const uint32_t* disp;
  const uint32_t* far;  // far guide: far_n + 1 entries
  uint64_t e_near, e_last;  // E[nnear - 1], E[K - 1]
  int32_t nnear, K;
  int32_t near_shift, far_shift;
  uint32_t far_n;
  __device__ __forceinline__ uint64_t w(int32_t k) const { return __ldg(&W[k]); }
  __device__ __forceinline__ uint32_t d(int32_t k) const {
    return k < nnear ? sD[k] : __ldg(&disp[k]);
  }
  __device__ __forceinline__ uint64_t e(int32_t k) const {
    return k < nnear ? sE[k] : __ldg(&E[k]);
  }
  // first k in [lo, K) with W[k] >= target, K if none.  Used where the walk's hazards are large, so that
  // the next candidate is mostly lo itself or near it: the bracket doubles from there (a binary search
  // of the whole list read it 15 times and more in global memory)
  __device__ __forceinline__ int32_t lower_bound(int32_t lo, uint64_t target) const {
    uint32_t a = (uint32_t)lo, b = a, step = 1;
    while (b < (uint32_t)K && __ldg(&W[b]) < target) {
      a = b + 1;
      b = a + step < (uint32_t)K ? a + step : (uint32_t)K;
      step *= 2;
    }
    while (a < b) {
      const uint32_t mid = (a + b) >> 1;
      if (__ldg(&W[mid]) >= target) b = mid; else a = mid + 1;
    }
    return (int32_t)a;
  }
  // first k with E[k] <= tb (E is non-increasing), K if none: between two guide entries.  A whole
  // binary search took 11 dependent shared-memory reads for a near candidate and 22 reads of the
  // list in global memory for a far one (5.8% of the candidates at T = 0.6 D, hence some lane of
  // most warps); the guides leave about two and four.
  __device__ __forceinline__ int32_t first_le(uint64_t tb) const {
    if (tb >= e_near) {
      const uint32_t q = (uint32_t)((kDecayStart - tb) >> near_shift);
      uint32_t a = sG[q], b = sG[q + 1];
      while (a < b) {
        const uint32_t mid = (a + b) >> 1;
        if (sE[mid] <= tb) b = mid; else a = mid + 1;
      }
      return (int32_t)a;
    }
    const uint64_t q64 = (e_near - tb) >> far_shift;
    const uint32_t q = q64 < far_n ? (uint32_t)q64 : far_n - 1;
    uint32_t a = __ldg(&far[q]), b = __ldg(&far[q + 1]);
    while (a < b) {
      const uint32_t mid = (a + b) >> 1;
      if (__ldg(&E[mid]) <= tb) b = mid; else a = mid + 1;
    }
    return (int32_t)a;
  }
};

// The block's copies of the list's head (every thread of the block calls it, then __syncthreads).
struct NearShared {
  uint64_t e[kNear];
  uint32_t d[kNear];
  uint16_t g[kNearGuide + 1];
};
__device__ __forceinline__ NearTable near_table(const Search& S, NearShared& sh) {
  const int32_t K = S.K, nnear = K < kNear ? K : kNear;
  for (int q = threadIdx.x; q < nnear; q += blockDim.x) {
    sh.e[q] = S.E[q];
    sh.d[q] = S.disp[q];
  }
  NearTable T{};
  T.K = K;
  if (K > 0) {
    for (int q = threadIdx.x; q <= kNearGuide; q += blockDim.x) sh.g[q] = S.near[q];
    const SearchHead h = *S.head;
    T = NearTable{sh.e,     sh.d,     sh.g,  S.W, S.E,          S.disp,      S.far,
                  h.e_near, h.e_last, nnear, K,   h.near_shift, h.far_shift, S.far_n};
  }
  return T;
}

// Exact re-evaluation of the next candidate: min { k > s : beta D 2^-58 (W_k - W_s) >= -ln u+ }.
// The table view comes by value (its address would put the caller's copy in local memory).
__device__ __noinline__ int32_t next_candidate_dd(const DevParams& P, const NearTable T, int32_t s,
                                                  uint64_t Ws, double up) {
  const dd ln2 = {P.ln2_hi, P.ln2_lo};
  const dd E = dd_neg(dd_log(dd_from(up), ln2));
  const dd tau = dd_ldexp(dd_div(E, two_prod(P.beta, P.D)), 58);
  uint32_t a = (uint32_t)(s + 1), b = (uint32_t)T.K;
  while (a < b) {
    const uint32_t mid = (a + b) >> 1;
    if (!dd_lt(dd_from_u64(T.w((int32_t)mid) - Ws), tau)) b = mid; else a = mid + 1;
  }
  return (int32_t)a;
}

// ceil(x) as an integer for finite x >= 0 (saturating at 2^64 - 1), from the bits of x with
// integer operations only (64-bit conversions would run on the FP64 pipe).
__device__ __forceinline__ uint64_t ceil_u64d(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  if (b == 0ull || (b >> 63)) return 0ull;
  const int ex = (int)((b >> 52) & 0x7FFu) - 1075;  // x = mant * 2^ex
  const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  if (ex >= 0) return ex >= 11 ? ~0ull : mant << ex;
  if (ex <= -54) return 1ull;  // 0 < x < 1
  const uint64_t q = mant >> (-ex);
  return q + ((q << (-ex)) != mant ? 1ull : 0ull);
}

// The candidate search with a logarithm, for what the decay table leaves open (targets below
// 2^-990 at very low temperatures, or next to a table value).
// tau = -ln(u+) / (beta D 2^-58) carries < 2^-48 relative error (log_np within kLogRelErr =
// 2^-49, fl(beta D), fl(2^58 / bD), one product); the candidate is certain when
// W_k - W_s >= tau (1 + 2^-46) and
// W_(k-1) - W_s < tau (1 - 2^-46), compared as integers (ceil of the bounds).
__device__ __noinline__ int32_t next_candidate(const DevParams& P, const NearTable T, int32_t s,
                                               uint64_t wE, unsigned& ghits) {
  const uint64_t Ws = s >= 0 ? T.w(s) : 0ull;
  const double up = u53pos(wE);
  const double tau = -log_np(up) * P.inv_bD58;
  const uint64_t rem = T.w(T.K - 1) - Ws;
  const uint64_t thr = ceil_u64d(tau);
  int32_t k = T.K;
  if (thr <= rem) k = T.lower_bound(s + 1, Ws + thr);
  // thr = ceil(tau): ceil(tau (1 + 2^-46)) <= thr + floor(thr 2^-46) + 1 = hi and
  // tau (1 - 2^-46) >= (thr - 1)(1 - 2^-46) >= thr - floor(thr 2^-46) - 2 = lo (saturating),
  // in integers: no FP64 instruction
  const uint64_t m46 = thr >> 46;
  const uint64_t hi = thr + m46 + 1 < thr ? ~0ull : thr + m46 + 1;  // >= hi: surely a candidate
  const uint64_t lo = thr > m46 + 2 ? thr - m46 - 2 : 0ull;         // < lo: surely not
  bool certain = true;
  if (k < T.K && T.w(k) - Ws < hi) certain = false;
  if (k - 1 > s && T.w(k - 1) - Ws >= lo) certain = false;
  if (certain) return k;
  ++ghits;
  return next_candidate_dd(P, T, s, Ws, up);
}

// ceil(x) as above for a float.
__device__ __forceinline__ uint64_t ceil_u64f(float x) {
  const uint32_t b = __float_as_uint(x);
  if (b == 0u || (b >> 31)) return 0ull;
  const int ex = (int)((b >> 23) & 0xFFu) - 150;  // x = mant * 2^ex
  const uint64_t mant = (uint64_t)((b & 0x7FFFFFu) | 0x800000u);
  if (ex >= 0) return ex >= 40 ? ~0ull : mant << ex;
  if (ex <= -25) return 1ull;  // 0 < x < 1
  const uint64_t q = mant >> (-ex);
  return q + ((q << (-ex)) != mant ? 1ull : 0ull);
}

// FP32 screen of that search (FP32-guarded form): E = -ln u+ as -log1pf(-(1 - u+)) above 1/2 (1 - u+ is
// an integer times 2^-53) and -logf(u+) below, relative error below 2^-20.5 (one input rounding, 4 ulp
// of the function); tau = E fl32(2^58 / bD) adds two roundings.  Margins inside 2^-18 fall through to
// the FP64 search.  Comparisons with W are made in integers.  Without it the FP32 form's switch at T =
// 0.02 D (L = 64) took 0.696 ms, with it 0.630 (T =
// 0.001 D: 3.01 and 2.54).
__device__ __noinline__ int32_t next_candidate_f32(const DevParams& P, const NearTable T, int32_t s,
                                                   uint64_t wE, unsigned& g32, unsigned& ghits) {
  const uint64_t Ws = s >= 0 ? T.w(s) : 0ull;
  const uint64_t m53 = wE >> 11;  // u+ = (m53 + 1) 2^-53
  const bool high = m53 >= (1ull << 52);
  const uint64_t m = high ? (1ull << 53) - 1ull - m53 : m53 + 1ull;  // <= 2^52
  const float v = __uint2float_rn((uint32_t)(m >> 20)) * 0x1p-33f +
                  __uint2float_rn((uint32_t)(m & 0xFFFFFu)) * 0x1p-53f;
  const float tau = -(high ? log1pf(-v) : logf(v)) * P.inv_bD58_f;
  const uint64_t rem = T.w(T.K - 1) - Ws;
  const uint64_t thr = ceil_u64f(tau);
  int32_t k = T.K;
  if (thr <= rem) k = T.lower_bound(s + 1, Ws + thr);
  // as in next_candidate, with 2^-18
  const uint64_t m18 = thr >> 18;
  const uint64_t hi = thr + m18 + 1 < thr ? ~0ull : thr + m18 + 1;
  const uint64_t lo = thr > m18 + 2 ? thr - m18 - 2 : 0ull;
  bool certain = tau < 0x1p62f;
  if (k < T.K && T.w(k) - Ws < hi) certain = false;
  if (k - 1 > s && T.w(k - 1) - Ws >= lo) certain = false;
  if (certain) return k;
  ++g32;
  return next_candidate(P, T, s, wE, ghits);
}

// Targets below 2^-990 take the search with a logarithm (the decay table's values there are not
// normal).
constexpr uint64_t kDecayMinBits = 0x0210000000000000ull;

// Candidate search without a logarithm.  With E*_m = exp(-beta D 2^-58 W_m) the next
// candidate min { k > s : beta D 2^-58 (W_k - W_s) >= -ln u+ } is min { k > s : E*_k <= u+ E*_s }
// (exp is increasing), searched on the table's bits: E_m within 2^-50 of E*_m, the target
// fl(u+ E_s) within 2^-49.9 of u+ E*_s.  Positive doubles order as their bit images, and 32
// units in the last place are at least 2^-48 relative, more than the combined error, so the
// candidate is certain when E_k's bits lie at least 32 below the target's and E_(k-1)'s at least
// 32 above; otherwise (or for a target below 2^-990) the search with the logarithm decides.
// Es carries the bits of E at the walk's last candidate and is advanced to the new one.
template <int PREC>
__device__ __forceinline__ int32_t next_candidate_e(const DevParams& P, const NearTable& T,
                                                    int32_t s, uint64_t& Es, uint64_t wE,
                                                    unsigned& g32, unsigned& ghits) {
  if (s >= T.K - 1 || !P.switching) return T.K;
  const uint64_t tb = (uint64_t)__double_as_longlong(u53pos(wE) * __longlong_as_double(Es));
  if (tb >= kDecayMinBits) {
    if (T.e_last >= tb + 32ull) return T.K;  // surely no candidate left: the walk ends
    const int32_t k = max(T.first_le(tb), s + 1);
    const uint64_t ek = k < T.K ? T.e(k) : 0ull;
    bool certain = true;
    if (k < T.K && ek + 32ull > tb) certain = false;
    if (k - 1 > s && T.e(k - 1) < tb + 32ull) certain = false;
    if (certain) {
      Es = ek;
      return k;
    }
  }
  const int32_t k = PREC == 1 ? next_candidate_f32(P, T, s, wE, g32, ghits)
                              : next_candidate(P, T, s, wE, ghits);
  if (k < T.K) Es = T.e(k);
  return k;
}

// Exact survival test u q < 1 - P_ij in double-double.  The spins come by value, so that the
// callers' spin copies stay in registers (an address passed to a function that is not inlined
// would put them in local memory on the fast path too).
__device__ __noinline__ bool survives_dd(const DevParams& P, double si0, double si1, double si2,
                                         double sj0, double sj1, double sj2, int32_t dx,
                                         int32_t dy, uint64_t A, double u1) {
  const double Si[3] = {si0, si1, si2}, Sj[3] = {sj0, sj1, sj2};
  const dd ln2 = {P.ln2_hi, P.ln2_lo};
  const int64_t r2 = (int64_t)dx * dx + (int64_t)dy * dy;
  const dd V = dd_pair_V(P.D, coupling_c(r2), (double)r2, Si, Sj, (double)dx, (double)dy);
  const dd Vm = dd_vmax(P.D, A);
  const dd b = dd_mul_d(dd_sub(V, Vm), P.beta);
  const dd a = dd_mul_d(Vm, 2.0 * P.beta);
  const dd pr = dd_neg(dd_expm1(b, ln2));
  const dd q = dd_neg(dd_expm1(dd_neg(a), ln2));
  return dd_lt(dd_mul_d(q, u1), pr);
}

// The integer hazard A_k of list element k (only the double-double tests need it).
__device__ __forceinline__ uint64_t hazard_of(const NearTable& T, int32_t k) {
  return T.w(k) - (k > 0 ? T.w(k - 1) : 0ull);
}

// Survival test u q < 1 - P_ij in float-float (df32.cuh): y = beta (Vmax - V) from the pair
// constants, 1 - P = 1 - e^-y; q as h + l within 2^-48 of the FP64 value, u within 2^-48.  The
// error of mu = (1 - P) - u q is below c0 = 2^-40 a1 (|dy|) plus 2^-31 (1 - P) plus 2^-43 q; the
// test is certain when |mu| exceeds four times that.  The FP64 form of it (23 FP64 instructions
// per candidate) kept the FP64 pipe 65% busy through the whole switch.
__device__ __forceinline__ bool survives_df(const DevParams& P, const PairDf& t, float2 q,
                                            const SpinDf& Si, const SpinDf& Sj, int32_t dx,
                                            const double* __restrict__ s, int64_t i, int64_t j,
                                            int32_t dy, const NearTable& T, int32_t k, uint64_t wU,
                                            unsigned& ghits) {
  const FieldDf g = df_field(t, dx < 0 ? -t.ax : t.ax, t.ay, Sj);
  df y = df_pair_y(t, g, Si);
  if (y.h > kYMin) {
    // e^-y is below 2^-144 from 100 on, where a1 2^-38 still bounds the error (y beyond the range of the
    // exponential went to double-double: every such candidate below about T = D / 2048)
    if (y.h > 100.f) y = {100.f, 0.f};
    const df pr = df_one_minus_exp_neg(y);
    const uint64_t m = wU >> 11;  // u = m 2^-53
    const df u = {(float)(uint32_t)(m >> 29) * 0x1p-24f,
                  (float)((uint32_t)m & 0x1FFFFFFFu) * 0x1p-53f};
    const df uq = df_mul(u, {q.x, q.y});
    const float mu = (pr.h - uq.h) + (pr.l - uq.l);
    const float lim = 0x1p-29f * pr.h + (0x1p-38f * t.a1h + 0x1p-41f * q.x);
    if (mu > lim) return true;
    if (mu < -lim) return false;
  }
  ++ghits;
  return survives_dd(P, s[i], s[P.N + i], s[2 * P.N + i], s[j], s[P.N + j], s[2 * P.N + j], dx, dy,
                     hazard_of(T, k), u53(wU));
}

// FP32 screen of the same test (FP32-guarded form): spins from the FP32 shadow
// (|dS| <= 2^-24 per component), table constants rounded to FP32, expm1f within 4 ulp.
// Falls through to the float-float test (and from there to double-double) inside the bound; only
// then are the FP64 spins of i and j read from the SoA array s.
__device__ __forceinline__ bool survives_fp32(const DevParams& P, float4 t32,
                                              const PairDf* __restrict__ pdf,
                                              const float2* __restrict__ qdf, int64_t tix,
                                              const float* Si32, const float* Sj32,
                                              const double* __restrict__ s, int64_t i, int64_t j,
                                              int32_t dx, int32_t dy, const NearTable& T,
                                              int32_t k, uint64_t wU, unsigned& g32,
                                              unsigned& ghits) {
  const float fr2 = (float)(dx * dx + dy * dy), fx = (float)dx, fy = (float)dy;
  // u truncated to 24 bits: 0 <= u - u24 < 2^-24, inside the 2^-19 q term of the bound
  const float u24 = __uint2float_rn((uint32_t)(wU >> 40)) * 0x1p-24f;
  const float ss = Si32[0] * Sj32[0] + Si32[1] * Sj32[1] + Si32[2] * Sj32[2];
  const float pa = Si32[0] * fx + Si32[1] * fy;
  const float pb = Sj32[0] * fx + Sj32[1] * fy;
  const float V = t32.x * (fr2 * ss - 3.0f * (pa * pb));
  const float beta = P.beta_f;
  const float b = beta * (V - t32.y);
  const float pr = -expm1f(b);
  const float q = t32.w;  // fl32 of the FP64 q: 2^-24 on top of its 4 ulp
  const float mu = pr - u24 * q;
  // |dV| <= 2^-17 Dc r^2 (shadow spins, FP32 products, constant rounding); beta and the
  // constants carry 2^-24 each; expm1f 4 ulp; generous factor 2.
  const float dV = 0x1p-17f * t32.x * fr2;
  const float B = 2.0f * (beta * (dV + 0x1p-22f * t32.y) + 0x1p-21f * fabsf(b) +
                          0x1p-19f * (fabsf(pr) + q) + 0x1p-21f * t32.z);
  if (mu > B) return true;
  if (mu < -B) return false;
  ++g32;
  const SpinDf Si = spin_df(s[i], s[P.N + i], s[2 * P.N + i], 0.0);
  const SpinDf Sj = spin_df(s[j], s[P.N + j], s[2 * P.N + j], 0.0);
  return survives_df(P, load32(pdf + tix), __ldg(qdf + tix), Si, Sj, dx, s, i, j, dy, T, k, wU,
                     ghits);
}

// Where a site writes its upper neighbours: kSlotCap slots of its own (row `id` of hslot), then
// an overflow list shared by all sites (entry: site id, j | flag).  indeg counts lower
// neighbours per (local) site.
struct SwitchOut {
  uint32_t* hslot;
  uint32_t* indeg;
  uint32_t* ovf;
  uint32_t ovf_cap;
  unsigned long long* ovf_n;
  int* status;
};

// One site's walk along its half-plane list: the candidate search of Sec. 2.1 with the state it
// carries from one candidate to the next, so that a thread can take the candidates one at a time
// (and take up another site when its list ends).
template <int PREC>
struct SiteWalk {
  uint32_t i;   // local site index (the Philox counter)
  uint32_t id;  // site id in the slots and the overflow list
  int32_t xi, yi;
  SpinDf Sd;       // FP64 form
  float Si32[3];   // FP32-screened form
  int32_t sidx;    // last candidate (-1 before the first)
  uint64_t Es;     // the bits of E at sidx
  uint32_t n;      // Philox blocks drawn (two candidates each)
  uint32_t n_out;
  bool nn0, nn1;
};

// The temperature-dependent tables by (|dx|, |dy|) and the spins that the survival tests read.
struct SwitchIn {
  const PairDf* pdf;
  const float2* qdf;
  const float4* xy32;
  const double* s;
  const float4* s32;  // FP32-guarded form
  const SpinDf* sd;   // FP64 form
};

__device__ __forceinline__ void switch_emit(const SwitchOut& o, uint32_t id, uint32_t& n_out,
                                            uint32_t jv) {
  if (n_out < (uint32_t)kSlotCap) {
    o.hslot[(size_t)id * kSlotCap + n_out] = jv;
  } else {
    const unsigned long long idx = atomicAdd(o.ovf_n, 1ull);
    if (idx < o.ovf_cap) {
      o.ovf[2 * idx] = id;
      o.ovf[2 * idx + 1] = jv;
    } else {
      set_status(o.status, kStatusCapacity);
    }
  }
  ++n_out;
  atomicAdd(&o.indeg[jv & kIndexMask], 1u);
}

template <int PREC>
__device__ __forceinline__ void walk_begin(const DevParams& P, const SwitchIn& in, uint32_t i,
                                           uint32_t id, SiteWalk<PREC>& a) {
  a.i = i;
  a.id = id;
  site_xy(i, P, a.xi, a.yi);
  if (PREC == 0) {
    a.Sd = load32(in.sd + i);
  } else {
    const float4 si = in.s32[i];
    a.Si32[0] = si.x;
    a.Si32[1] = si.y;
    a.Si32[2] = si.z;
  }
  a.sidx = -1;
  a.Es = kDecayStart;
  a.n = 0;
  a.n_out = 0;
  a.nn0 = false;
  a.nn1 = false;
}

// Draws the next two candidates of the walk (one Philox block) and tests the survival of those
// that lie on the lattice (emitting the pairs that survive).  Returns false once the list is
// exhausted.  Two per call, because a lane draws a block for every second candidate: with one per
// call the lanes of a warp stood at both parities and the block's 280 instructions were issued at
// every call for half of them.
template <int PREC>
__device__ __forceinline__ bool walk_step(const DevParams& P, const NearTable& T,
                                          const SwitchIn& in, uint32_t epoch, int32_t mnn0,
                                          int32_t mnn1, const SwitchOut& o, SiteWalk<PREC>& a,
                                          unsigned& n_dip, unsigned& ghits, unsigned& g32) {
  W4 w = philox((uint64_t)a.i, epoch, (uint64_t)a.n, kTagSwitch, P.key0, P.key1);
  ++a.n;
  bool more = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int32_t k = more ? next_candidate_e<PREC>(P, T, a.sidx, a.Es, w.w[0], g32, ghits) : T.K;
    more = k < T.K;
    const uint64_t wU = w.w[1];
    w.w[0] = w.w[2];
    w.w[1] = w.w[3];
    if (!more) continue;
    a.sidx = k;
    const uint32_t d = T.d(k);
    const int32_t dx = (int16_t)(d & 0xFFFFu), dy = (int32_t)(d >> 16);
    const int32_t xj = a.xi + dx, yj = a.yi + dy;
    if (xj < 0 || xj >= P.Lx || yj >= P.Ly) continue;
    const uint32_t j = (uint32_t)xj + (uint32_t)P.Lx * (uint32_t)yj;
    const int64_t tix = (int64_t)(dx < 0 ? -dx : dx) + (int64_t)P.Lx * dy;
    bool surv;
    if (PREC == 1) {
      const float4 sj = in.s32[j];
      const float Sj32[3] = {sj.x, sj.y, sj.z};
      surv = survives_fp32(P, __ldg(&in.xy32[tix]), in.pdf, in.qdf, tix, a.Si32, Sj32, in.s,
                           (int64_t)a.i, (int64_t)j, dx, dy, T, k, wU, g32, ghits);
    } else {
      surv = survives_df(P, load32(in.pdf + tix), __ldg(&in.qdf[tix]), a.Sd, load32(in.sd + j), dx,
                         in.s, (int64_t)a.i, (int64_t)j, dy, T, k, wU, ghits);
    }
    if (surv) {
      switch_emit(o, a.id, a.n_out, j);
      ++n_dip;
      if (k == mnn0) a.nn0 = true;
      if (k == mnn1) a.nn1 = true;
    }
  }
  return more;
}

// Ends the walk: exchange bonds that the dipolar switch did not keep join the colouring graph.
// Returns the number of upper neighbours written (dipolar survivors plus exchange-only bonds).
template <int PREC>
__device__ __forceinline__ uint32_t walk_end(const DevParams& P, int32_t mnn0, int32_t mnn1,
                                             const SwitchOut& o, SiteWalk<PREC>& a) {
  if (P.J != 0.0) {
    if (mnn0 >= 0 && !a.nn0 && a.xi + 1 < P.Lx) switch_emit(o, a.id, a.n_out, (a.i + 1) | kExchOnly);
    if (mnn1 >= 0 && !a.nn1 && a.yi + 1 < P.Ly)
      switch_emit(o, a.id, a.n_out, (a.i + (uint32_t)P.Lx) | kExchOnly);
  }
  return a.n_out;
}

// Switches the half-plane pairs of the sites below `end` that the calling warp claims, 32 at a time,
// from *next (local indices; site i writes slots id0 + i).  kRefill: a lane whose walk ends takes up
// the next claimed site at once, so that the lanes of a warp stay busy although the number of
// candidates differs from site to site (Poisson, mean about 14 at T = 0.6D); else the warp claims
// again once all its lanes are done.  One lattice (parameters in constant memory) is faster with it
// (switch phase at L = 2304 2.96 against 3.14 ms), the batch, whose parameters are read from shared
// memory at every step, without (64 replicas 2.45 against 3.10 ms).  Returns upper neighbours written.
template <int PREC, bool kRefill>
__device__ __forceinline__ unsigned switch_range(const DevParams& P, const NearTable& T,
                                                 const SwitchIn& in, uint32_t epoch, int32_t mnn0,
                                                 int32_t mnn1, unsigned* next, uint32_t end,
                                                 uint32_t id0, uint32_t* __restrict__ hcnt,
                                                 const SwitchOut& o, unsigned& n_dip,
                                                 unsigned& ghits, unsigned& g32) {
  const unsigned lane = threadIdx.x & 31u;
  unsigned n_half = 0;
  SiteWalk<PREC> a;
  if (!kRefill) {
    for (;;) {
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(next, 32u);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base >= end) return n_half;
      const uint32_t i = base + lane;
      if (i < end) {
        walk_begin<PREC>(P, in, i, id0 + i, a);
        while (walk_step<PREC>(P, T, in, epoch, mnn0, mnn1, o, a, n_dip, ghits, g32)) {
        }
        const uint32_t n_out = walk_end<PREC>(P, mnn0, mnn1, o, a);
        hcnt[a.id] = n_out;
        n_half += n_out;
      }
      __syncwarp();
    }
  }
  const unsigned below = (1u << lane) - 1u;
  bool active = false, drained = false;  // drained, pool and pool_n are warp-uniform
  uint32_t pool = 0, pool_n = 0;
  for (;;) {
    unsigned need = __ballot_sync(0xffffffffu, !active);
    while (need != 0u && !drained) {
      if (pool_n == 0u) {
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(next, 32u);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= end) {
          drained = true;
          break;
        }
        pool = base;
        pool_n = min(32u, end - base);
      }
      const uint32_t take = min((uint32_t)__popc(need), pool_n);
      const uint32_t rank = (uint32_t)__popc(need & below);
      if (!active && rank < take) {
        walk_begin<PREC>(P, in, pool + rank, id0 + pool + rank, a);
        active = true;
      }
      pool += take;
      pool_n -= take;
      need = __ballot_sync(0xffffffffu, !active);
    }
    const unsigned act = __ballot_sync(0xffffffffu, active);
    if (act == 0u) break;
    if (active && !walk_step<PREC>(P, T, in, epoch, mnn0, mnn1, o, a, n_dip, ghits, g32)) {
      const uint32_t n_out = walk_end<PREC>(P, mnn0, mnn1, o, a);
      hcnt[a.id] = n_out;
      n_half += n_out;
      active = false;
    }
  }
  return n_half;
}

// End of site i's group (see RowFill): neighbours below it from above i, and from below i those i is
// one of for, are near.
__device__ __forceinline__ uint32_t near_end(const RowFill& F, uint32_t i) {
  return F.group ? (i / F.group + 1) * F.group : 0u;
}
// The next place in site i's row.
__device__ __forceinline__ uint32_t row_place(const RowFill& F, bool near,
                                              const uint32_t* __restrict__ row_ptr,
                                              uint32_t* __restrict__ cur, uint32_t i) {
  const uint32_t base = row_ptr[near ? i + 1 : i];
  const uint32_t at = atomicAdd(&cur[i], near ? 0x10000u : 1u);
  return near ? base - 1 - (at >> 16) : base + (at & F.mask);
}
// The places of the overflow half-edge i -> jv in rows i and j.
__device__ __forceinline__ void fill_overflow(const RowFill& F, uint32_t i, uint32_t jv,
                                              const uint32_t* __restrict__ row_ptr,
                                              const uint32_t* __restrict__ indeg, uint32_t* hcnt,
                                              uint32_t* __restrict__ cur, uint32_t* __restrict__ col) {
  const uint32_t j = jv & kIndexMask;
  const bool near = j < near_end(F, i);
  // (a split row's larger neighbours beyond the slots: places hcnt - 1 down to kSlotCap of that part)
  const uint32_t at = F.split ? row_ptr[i] + indeg[i] + atomicSub(&hcnt[i], 1u) - 1u
                              : row_place(F, near, row_ptr, cur, i);
  col[at] = jv;
  col[row_place(F, near, row_ptr, cur, j)] = i | (jv & kExchOnly);
}

// Every surviving half-edge (i, j) of site i's slots goes into rows i and j (see RowFill; indices and
// arrays of one lattice): eight half-edges at a time, whose slot and row-pointer loads, atomics and
// stores are each issued together (the atomics' returns were the chain).
__device__ __forceinline__ void fill_rows(const RowFill& F, uint32_t i,
                                          const uint32_t* __restrict__ slot, uint32_t hcnt,
                                          const uint32_t* __restrict__ indeg,
                                          const uint32_t* __restrict__ row_ptr,
                                          uint32_t* __restrict__ cur, uint32_t* __restrict__ col) {
  const uint32_t n = min(hcnt, (uint32_t)kSlotCap);
  const uint32_t end = near_end(F, i);
  constexpr uint32_t kB = 8;
  for (uint32_t q0 = 0; q0 < n; q0 += kB) {
    uint32_t jv[kB], base[kB], at[kB];
    uint32_t nn = 0;
#pragma unroll
    for (uint32_t a = 0; a < kB; ++a) jv[a] = q0 + a < n ? slot[q0 + a] : kIndexMask;
#pragma unroll
    for (uint32_t a = 0; a < kB; ++a) {
      const uint32_t j = jv[a] & kIndexMask;
      const bool on = q0 + a < n, near = on && j < end;
      base[a] = on ? row_ptr[near ? j + 1 : j] : 0u;
      nn += near ? 1u : 0u;
    }
    uint32_t own = F.split ? indeg[i] + q0
                           : atomicAdd(&cur[i], (min(n - q0, kB) - nn) | (nn << 16));
#pragma unroll
    for (uint32_t a = 0; a < kB; ++a) {
      const uint32_t j = jv[a] & kIndexMask;
      at[a] = q0 + a < n ? atomicAdd(&cur[j], j < end ? 0x10000u : 1u) : 0u;
    }
    const uint32_t b = row_ptr[i], e = row_ptr[i + 1];
#pragma unroll
    for (uint32_t a = 0; a < kB; ++a) {
      if (q0 + a >= n) continue;
      const bool near = (jv[a] & kIndexMask) < end;
      col[near ? e - 1 - (own >> 16) : b + (own & F.mask)] = jv[a];
      own += near ? 0x10000u : 1u;
      col[near ? base[a] - 1 - (at[a] >> 16) : base[a] + (at[a] & F.mask)] = i | (jv[a] & kExchOnly);
    }
  }
}

}  // namespace
}  // namespace sco
