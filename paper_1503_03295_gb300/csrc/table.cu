// table.cu -- the translation-invariant coupling table, built on the device.
//
// Every unordered pair of the open lattice is (i, i + d) for one d of the half plane
// {dy > 0, |dx| < Lx} u {dy = 0, 0 < dx < Lx}.  The list is sorted by (r^2, dy, dx) with a
// stable counting sort on r^2 (rows are placed in increasing dy, and inside a row the
// negative dx before the positive one), each element carries the integer hazard
// A(r^2) > 2^60 / r^3 of its pair (V_max = D A 2^-59 >= 2D / r^3, Sec. 2.1), and W is the
// inclusive prefix of A.  A second table indexed by (|dx|, |dy|) holds fl(D c(r^2)) and
// V_max for the pair-energy evaluations of the switch and sweep kernels.
#include <cstdint>

#include "sco_internal.h"

namespace sco {

namespace {

__device__ __forceinline__ void disp_of_q(int64_t q, int32_t Lx, int32_t& dx, int32_t& dy) {
  if (q < Lx - 1) {
    dx = (int32_t)q + 1;
    dy = 0;
    return;
  }
  const int64_t r = q - (Lx - 1);
  const int64_t w = 2 * (int64_t)Lx - 1;
  dy = (int32_t)(r / w) + 1;
  dx = (int32_t)(r % w) - (Lx - 1);
}

__global__ void k_r2_count(int32_t Lx, int64_t K, uint32_t* __restrict__ cnt) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= K) return;
  int32_t dx, dy;
  disp_of_q(q, Lx, dx, dy);
  atomicAdd(&cnt[(int64_t)dx * dx + (int64_t)dy * dy], 1u);
}

// One block walks the rows dy = 0..Ly-1 in order.  Inside a row the values |dx| are
// distinct, hence so are the r^2, so the threads of a row never touch the same bucket.
__global__ void __launch_bounds__(1024) k_order(int32_t Lx, int32_t Ly,
                                                const uint32_t* __restrict__ start,
                                                uint32_t* __restrict__ seen,
                                                uint32_t* __restrict__ disp) {
  for (int32_t dy = 0; dy < Ly; ++dy) {
    for (int32_t ax = threadIdx.x; ax < Lx; ax += blockDim.x) {
      if (dy == 0 && ax == 0) continue;
      const int64_t r2 = (int64_t)ax * ax + (int64_t)dy * dy;
      uint32_t m = start[r2] + seen[r2];
      uint32_t n = 0;
      if (dy > 0 && ax > 0) {  // (-ax, dy) precedes (ax, dy)
        disp[m++] = ((uint32_t)(uint16_t)(int16_t)(-ax)) | ((uint32_t)dy << 16);
        ++n;
      }
      disp[m] = ((uint32_t)(uint16_t)(int16_t)ax) | ((uint32_t)dy << 16);
      ++n;
      seen[r2] += n;
    }
    __syncthreads();
  }
}

__global__ void k_hazard(int64_t K, const uint32_t* __restrict__ disp, uint64_t* __restrict__ A) {
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (m >= K) return;
  const uint32_t d = disp[m];
  const int32_t dx = (int16_t)(d & 0xFFFFu), dy = (int32_t)(d >> 16);
  A[m] = hazard_A((int64_t)dx * dx + (int64_t)dy * dy);
}

// Sweep constants of a pair at (|dx|, |dy|).  FP64 (Sw64): the field of S_j on site i scaled
// by beta, f = a1 S_j - (S_j . a3 d) d with a1 = fl(beta fl(Dc r^2)) and a3 d = fl(beta fl(3 Dc)) d,
// so x = beta V - fl(beta Vmax) = S_i . f - bvm; c0 bounds the part of |x error| that does not
// scale with |x|: |beta dV| <= 2^-46 beta Dc r^2 (FP64 products, the rounded beta-scaled
// constants) plus 2^-51 beta Vmax (fl(beta Vmax)), plus 2^-52 (2 beta Vmax) for the rounding of
// x itself (|x| <= 2 beta Vmax).
__global__ void k_xy(int32_t Lx, int32_t Ly, double D, double beta, double2* __restrict__ xy,
                     float2* __restrict__ qdf, float4* __restrict__ xy32,
                     Sw64* __restrict__ sw64, float4* __restrict__ sw32,
                     PairDf* __restrict__ pdf) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= (int64_t)Lx * Ly) return;
  const int64_t ax = q % Lx, ay = q / Lx;
  const int64_t r2 = ax * ax + ay * ay;
  double dc = 0.0, vm = 0.0;
  if (r2 > 0) {
    dc = __dmul_rn(D, coupling_c(r2));
    vm = __dmul_rn(__dmul_rn(D, (double)hazard_A(r2)), 0x1p-59);
  }
  const double a = (2.0 * beta) * vm;
  const double cq = -expm1(-a);
  xy[q] = make_double2(dc, vm);
  const df dq = df_split_const(cq);
  qdf[q] = make_float2(dq.h, dq.l);
  xy32[q] = make_float4((float)dc, (float)vm, (float)a, (float)cq);
  const double a1 = dc * (double)r2, a3 = 3.0 * dc, bvm = beta * vm;
  const double a3b = beta * a3;
  const double c64 = beta * (0x1p-46 * dc * (double)r2) + 0x1p-51 * bvm + 0x1p-52 * (2.0 * bvm);
  Sw64 t;
  t.a1 = beta * a1;
  t.a3x = a3b * (double)ax;
  t.a3y = a3b * (double)ay;
  t.ax = (double)ax;
  t.ay = (double)ay;
  t.bvm = bvm;
  t.c0 = c64 * (1.0 + 0x1p-20);
  sw64[q] = t;
  const df d1 = df_split_const(t.a1), d3 = df_split_const(a3b), dv = df_split_const(bvm);
  pdf[q] = PairDf{d1.h, d1.l, d3.h, d3.l, dv.h, dv.l, (float)ax, (float)ay};
  sw32[q] = make_float4((float)t.a1, (float)a3b, (float)bvm, 0.f);
}

// E_m = exp(-beta D 2^-58 W_m) as bits: the candidate process of the switch has rate
// beta D A_m 2^-58 per element, so E_m is the probability of passing elements 0..m without a
// candidate.  The exponent is formed exactly to double-double (beta D as an exact product, W_m split
// into two exact doubles) and E = exp(-hi) (1 - lo); with CUDA's exp taken at 4 ulp E_m lies within
// 2^-50 of its exact value (relative); below e^-690 (< 2^-995) it is stored as +0, which the
// search treats as below every target it accepts (targets under 2^-990 take the exact path).
__global__ void k_decay(int64_t K, double beta, double D, const uint64_t* __restrict__ W,
                        uint64_t* __restrict__ Eb) {
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (m >= K) return;
  const uint64_t w = W[m];
  const dd wd = dd_add(dd_from((double)(w >> 32) * 0x1p32), dd_from((double)(w & 0xFFFFFFFFull)));
  const dd a = dd_ldexp(dd_mul(two_prod(beta, D), wd), -58);
  double e = 0.0;
  if (a.hi < 690.0) {
    e = exp(-a.hi);
    e = fma(-a.lo, e, e);
  }
  Eb[m] = (uint64_t)__double_as_longlong(e);
}

// Both guides (see Search).  The cells' bounds fall with the cell number as E does with the element,
// so element m is the first at or below the bounds of the cells in (cell of E_(m-1), cell of E_m]:
// each element writes its own, and one thread past the list the rest (a binary search per cell took
// 20 us for a list of 32,000).  E is rounded: where neighbours differ by less than its error (beta D
// below about 1e-11) an entry may lie a few units above the one before it, or above the top of its
// guide.  The cells are therefore clamped to the guide; which of two such entries a cell then names is
// settled by the search's own margin of 32 units.
__host__ __device__ inline uint64_t guide_cell(uint64_t top, uint64_t e, int shift, uint64_t n) {
  if (e >= top) return 0;
  const uint64_t q = (top - e) >> shift;
  return q < n ? q : n;
}
// the smallest shift that leaves fewer than n cells (n a power of two) from top down to bottom
__host__ __device__ inline int guide_shift(uint64_t top, uint64_t bottom, uint64_t n) {
  if (top <= bottom) return 0;
#ifdef __CUDA_ARCH__
  const int s = __clzll((long long)n) - __clzll((long long)(top - bottom)) + 1;
#else
  const int s = __builtin_clzll(n) - __builtin_clzll(top - bottom) + 1;
#endif
  return s > 0 ? s : 0;
}
struct GuideRange {
  int64_t first, last;  // cells that an element writes (none: last < first)
};
// element m of the part [m0, m1) of the list, whose last one writes every remaining cell
__host__ __device__ inline GuideRange guide_range(const uint64_t* E, int64_t m, int64_t m0, int64_t m1,
                                                  uint64_t top, int shift, uint64_t n) {
  return {m > m0 ? (int64_t)guide_cell(top, E[m - 1], shift, n) + 1 : 0,
          m == m1 - 1 ? (int64_t)n : (int64_t)guide_cell(top, E[m], shift, n)};
}
__global__ void k_guide(int64_t K, uint32_t far_n, const uint64_t* __restrict__ Eb,
                        SearchHead* __restrict__ head, uint16_t* __restrict__ near_g,
                        uint32_t* __restrict__ far_g) {
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (m > K) return;
  const int64_t nnear = K < kNear ? K : kNear;
  SearchHead h;
  h.e_near = Eb[nnear - 1];
  h.e_last = Eb[K - 1];
  h.near_shift = guide_shift(kDecayStart, h.e_near, kNearGuide);
  h.far_shift = guide_shift(h.e_near, h.e_last, far_n);
  if (m == 0) *head = h;
  if (m < nnear) {
    const GuideRange r = guide_range(Eb, m, 0, nnear, kDecayStart, h.near_shift, kNearGuide);
    for (int64_t q = r.first; q <= r.last; ++q) near_g[q] = (uint16_t)m;
  }
  if (m >= nnear) {
    const GuideRange r = guide_range(Eb, m, nnear, K + 1, h.e_near, h.far_shift, far_n);
    for (int64_t q = r.first; q <= r.last; ++q) far_g[q] = (uint32_t)m;
  }
}

}  // namespace

cudaError_t table_build_xy(const DevParams& P, Table& t, const Table& list, cudaStream_t s,
                           int64_t* launches) {
  const int64_t nxy = (int64_t)P.Lx * P.Ly, K = list.K;
  t.far_n = 64;  // one cell per 16 elements of the list, up to kFarGuide
  while (t.far_n < kFarGuide && (int64_t)t.far_n * 16 < K) t.far_n *= 2;
  // one allocation for all of them (a batch builds them per replica)
  size_t bytes = 0;
  auto place = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) / 256 * 256;
    return at;
  };
  const size_t o_xy = place(nxy * sizeof(double2)), o_xy32 = place(nxy * sizeof(float4)),
               o_q = place(nxy * sizeof(float2)), o_sw64 = place(nxy * sizeof(Sw64)),
               o_sw32 = place(nxy * sizeof(float4)), o_pdf = place(nxy * sizeof(PairDf)),
               o_e = place(K * sizeof(uint64_t)), o_head = place(sizeof(SearchHead)),
               o_near = place((kNearGuide + 1) * sizeof(uint16_t)),
               o_far = place((t.far_n + 1) * sizeof(uint32_t));
  if (t.pool_bytes < bytes) {
    table_free_xy(t);
    const cudaError_t e = cudaMalloc(&t.pool, bytes);
    if (e != cudaSuccess) return e;
    t.pool_bytes = bytes;
  }
  char* p = static_cast<char*>(t.pool);
  t.xy = reinterpret_cast<double2*>(p + o_xy);
  t.xy32 = reinterpret_cast<float4*>(p + o_xy32);
  t.qdf = reinterpret_cast<float2*>(p + o_q);
  t.sw64 = reinterpret_cast<Sw64*>(p + o_sw64);
  t.sw32 = reinterpret_cast<float4*>(p + o_sw32);
  t.pdf = reinterpret_cast<PairDf*>(p + o_pdf);
  t.Ebits = reinterpret_cast<uint64_t*>(p + o_e);
  t.head = reinterpret_cast<SearchHead*>(p + o_head);
  t.near_g = reinterpret_cast<uint16_t*>(p + o_near);
  t.far_g = reinterpret_cast<uint32_t*>(p + o_far);
  k_xy<<<(unsigned)((nxy + 255) / 256), 256, 0, s>>>(P.Lx, P.Ly, P.D, P.beta, t.xy, t.qdf,
                                                      t.xy32, t.sw64, t.sw32, t.pdf);
  ++*launches;
  if (K > 0) {
    k_decay<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(K, P.beta, P.D, list.W, t.Ebits);
    k_guide<<<(unsigned)((K + 1 + 255) / 256), 256, 0, s>>>(K, t.far_n, t.Ebits, t.head, t.near_g,
                                                            t.far_g);
    *launches += 2;
  }
  return cudaGetLastError();
}

cudaError_t table_build_list(const DevParams& P, Table& t, cudaStream_t s, int64_t* launches) {
  cudaError_t e;
  const int64_t K = P.K;
  t.K = K;
  if ((e = cudaMalloc(&t.disp, (K > 0 ? K : 1) * sizeof(uint32_t))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&t.W, (K > 0 ? K : 1) * sizeof(uint64_t))) != cudaSuccess) return e;
  if (K == 0) return cudaGetLastError();
  const int64_t R2 = (int64_t)(P.Lx - 1) * (P.Lx - 1) + (int64_t)(P.Ly - 1) * (P.Ly - 1);
  uint32_t *cnt = nullptr, *start = nullptr;
  uint64_t *A = nullptr, *tmp = nullptr;
  const int64_t ns = (R2 + 2 > K ? R2 + 2 : K);
  e = cudaMalloc(&cnt, (R2 + 2) * sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaMalloc(&start, (R2 + 2) * sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaMalloc(&A, K * sizeof(uint64_t));
  if (e == cudaSuccess) e = cudaMalloc(&tmp, scan_tmp_bytes(ns));
  if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (R2 + 2) * sizeof(uint32_t), s);
  if (e == cudaSuccess) {
    k_r2_count<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(P.Lx, K, cnt);
    ++*launches;
    e = scan_excl_u32(cnt, start, R2 + 1, tmp, nullptr, s, launches);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (R2 + 2) * sizeof(uint32_t), s);
  if (e == cudaSuccess) {
    k_order<<<1, 1024, 0, s>>>(P.Lx, P.Ly, start, cnt, t.disp);
    ++*launches;
    k_hazard<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(K, t.disp, A);
    ++*launches;
    e = scan_incl_u64(A, t.W, K, tmp, nullptr, s, launches);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(cnt);
  cudaFree(start);
  cudaFree(A);
  cudaFree(tmp);
  if (e != cudaSuccess) return e;
  // table index of the two nearest-neighbour displacements (1,0) and (0,1)
  uint32_t head[2] = {0, 0};
  const int nh = K < 2 ? (int)K : 2;
  if ((e = cudaMemcpy(head, t.disp, nh * sizeof(uint32_t), cudaMemcpyDeviceToHost)) != cudaSuccess)
    return e;
  for (int q = 0; q < nh; ++q) {
    if (head[q] == 1u) t.m_nn[0] = q;
    if (head[q] == (1u << 16)) t.m_nn[1] = q;
  }
  return cudaGetLastError();
}

cudaError_t table_build(const DevParams& P, Table& t, cudaStream_t s, int64_t* launches) {
  cudaError_t e = table_build_list(P, t, s, launches);
  if (e == cudaSuccess) e = table_build_xy(P, t, t, s, launches);
  return e;
}

void table_free_xy(Table& t) {
  cudaFree(t.pool);
  t.pool = nullptr;
  t.pool_bytes = 0;
  t.xy = nullptr;
  t.qdf = nullptr;
  t.xy32 = nullptr;
  t.sw64 = nullptr;
  t.sw32 = nullptr;
  t.pdf = nullptr;
  t.Ebits = nullptr;
  t.head = nullptr;
  t.near_g = nullptr;
  t.far_g = nullptr;
}

void table_free(Table& t) {
  cudaFree(t.disp);
  cudaFree(t.W);
  table_free_xy(t);
  t = Table();
}

}  // namespace sco
