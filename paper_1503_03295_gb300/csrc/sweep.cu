// sweep.cu -- step (B) of Sec. 2.1 / step (3) of Fig. 1 for one lattice: Metropolis
// updates of all sites of one colour class at a time (one launch per colour), with the
// undecided sites settled afterwards by one warp each.  Sites of one colour share no pair,
// so they update independently.  The per-site decision is in sweep_dev.cuh.
#include <cstdint>

#include "sweep_dev.cuh"

namespace sco {

namespace {

// Draws the proposal of every site for MC step `step` (see take_proposal); propd (FP64 form): the
// same in float-float, with u (u_h = -1: no move).
__global__ void __launch_bounds__(256) k_propose(const DevParams P, uint64_t step,
                                                 double4_32a* __restrict__ prop,
                                                 SpinDf* __restrict__ propd) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  SiteCtx c;
  c.i = i;
  const bool ok = propose(P, c, step);
  prop[i] = ok ? make_double4_32a(c.Sn[0], c.Sn[1], c.Sn[2], c.u)
               : make_double4_32a(0.0, 0.0, 1.0, -1.0);
  if (propd) {
    SpinDf d = spin_df(c.Sn[0], c.Sn[1], c.Sn[2], c.u);
    if (!ok) d.u_h = -1.f;
    propd[i] = d;
  }
}

// One site's decision in FP64 then double-double by a whole warp, for the sites that the
// float-float decision leaves open (about one in 10^6): a function of its own, so that its
// registers stay out of the sweep.
__device__ __noinline__ bool settle_site(const DevParams& P, uint32_t i,
                                         const Sw64* __restrict__ sw, const double* s,
                                         const uint32_t* __restrict__ row_ptr,
                                         const uint32_t* __restrict__ col,
                                         const double4_32a* __restrict__ prop, int lane,
                                         unsigned& ndd) {
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

struct SweepArgs {
  const PairDf* pdf;
  const Sw64* sw;
  double* s;
  SpinDf* sd;
  const uint32_t* row_ptr;
  const uint32_t* col;
  const uint32_t* perm;
  const uint32_t* off;
  const double4_32a* prop;
  const SpinDf* propd;
  uint8_t* acc;
  DevCounters* cnt;
};

// The n sites of the class at perm[b], kG lanes per site, grid-stride by warps.
template <int kG>
__device__ __forceinline__ void sweep_class(const DevParams& P, const SweepArgs& A, uint32_t b,
                                            uint32_t n, unsigned& ndd) {
  constexpr uint32_t kSites = 32 / kG;  // per warp
  const int lane = threadIdx.x & 31, sub = lane % kG;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t step = ((gridDim.x * blockDim.x) >> 5) * kSites;
  for (uint32_t q = warp * kSites; q < n; q += step) {
    const uint32_t idx = q + lane / kG;
    uint32_t i = 0, e0 = 0, e1 = 0;
    int d = 0;
    SpinDf S, N;
    N.u_h = -1.f;
    if (idx < n) {
      i = A.perm[b + idx];
      N = load32(A.propd + i);
      if (N.u_h >= 0.f) {
        e0 = A.row_ptr[i];
        e1 = A.row_ptr[i + 1];
        S = load32(A.sd + i);
      }
    }
    int32_t xi, yi;
    site_xy(i, P, xi, yi);
    d = accept_df<kG>(P, xi, yi, S, N, A.pdf, A.sd, A.col, e0, e1, i, sub);
    const bool mine = sub == 0 && idx < n;
    if (!mine || N.u_h < 0.f) d = 0;
    for (unsigned open = __ballot_sync(0xffffffffu, d == 2); open != 0; open &= open - 1) {
      const int src = __ffs(open) - 1;
      const bool r = settle_site(P, __shfl_sync(0xffffffffu, i, src), A.sw, A.s, A.row_ptr, A.col,
                                 A.prop, lane, ndd);
      if (lane == src) d = r ? 1 : 0;
    }
    if (mine) {
      if (d == 1) {
        const double4_32a v = A.prop[i];
        A.s[i] = v.x;
        A.s[P.N + i] = v.y;
        A.s[2 * P.N + i] = v.z;
        A.sd[i] = N;
      }
      A.acc[i] = d == 1 ? 1 : 0;
    }
  }
}

// FP64 form: the sites of one colour, decided in float-float (accept_df); undecided ones settled
// at once by their warp.  Bound by FP32 issue and the neighbour gathers: 2.20 ms per step at
// L = 2304, T = 0.6 D (k = 17.8) where the FP64 evaluation with its cache of pair terms took 7.10
// (64 registers and 8 blocks per SM; 80 and 6: 2.34, 96 and 5: 2.59).
//
// Lanes per site: 2 while the class gives every second lane of the grid a site (one lane per site
// took 2.37 ms at L = 2304, four 2.28; two lanes read a row in half the dependent steps), 8 and 32
// below, where the class would leave the grid idle and a row's serial chain sets the time (L = 256,
// 8192 sites in the largest classes: 0.230 ms per step with 8 and 32, 0.256 with 4 and 16).
__global__ void __launch_bounds__(128, 8) k_sweep_df(const __grid_constant__ DevParams P,
                                                     const __grid_constant__ SweepArgs A,
                                                     uint32_t colour) {
  const uint32_t b = A.off[colour], n = A.off[colour + 1] - b;
  const uint32_t nth = gridDim.x * blockDim.x;
  unsigned ndd = 0;
  if (n >= nth / 2) sweep_class<2>(P, A, b, n, ndd);
  else if (n >= nth / 32) sweep_class<8>(P, A, b, n, ndd);
  else sweep_class<32>(P, A, b, n, ndd);
  if ((threadIdx.x & 31) == 0 && ndd) atomicAdd(&A.cnt->guard_fp64, (unsigned long long)ndd);
}

// FP32-guarded form: one thread per site of the class.  A site whose decision stays inside the
// error bound is appended to the deferred list of the colour and settled by k_resolve (one warp
// per site), so that no thread of this kernel runs the FP64 / double-double evaluations.
__global__ void __launch_bounds__(128, 8) k_sweep32(const DevParams P,
                                                    const float4* __restrict__ sw32,
                                                    double* __restrict__ s,
                                                    float4* __restrict__ s32,
                                                    const uint32_t* __restrict__ row_ptr,
                                                    const uint32_t* __restrict__ col,
                                                    const uint32_t* __restrict__ perm,
                                                    const uint32_t* __restrict__ off,
                                                    uint32_t colour,
                                                    const double4_32a* __restrict__ prop,
                                                    uint8_t* __restrict__ acc,
                                                    uint32_t* __restrict__ defer,
                                                    uint32_t* __restrict__ dcnt,
                                                    DevCounters* __restrict__ cnt) {
  const uint32_t b = off[colour], e = off[colour + 1];
  unsigned long long nd = 0;
  for (uint32_t idx = b + blockIdx.x * blockDim.x + threadIdx.x; idx < e;
       idx += gridDim.x * blockDim.x) {
    SiteCtx c;
    load_site(P, c, perm[idx], s);
    if (!take_proposal(c, prop)) {
      acc[c.i] = 0;
      continue;
    }
    const int d = c.u != 0.0 ? accept_fp32(P, c, sw32, s32, row_ptr, col) : 1;
    if (d == 2) {
      defer[b + atomicAdd(&dcnt[colour], 1u)] = (uint32_t)c.i;
      ++nd;
      continue;
    }
    write_site(P, c, d == 1, s, s32, acc);
  }
  nd = warp_sum_u64(nd);
  if ((threadIdx.x & 31) == 0 && nd) atomicAdd(&cnt->guard_fp32, nd);
}

// Settles the deferred sites of a colour (FP32-guarded form): one warp per site, FP64 then
// double-double.
__global__ void __launch_bounds__(128) k_resolve(const __grid_constant__ DevParams P,
                                                 const Sw64* __restrict__ sw,
                                                 double* __restrict__ s, float4* __restrict__ s32,
                                                 const uint32_t* __restrict__ row_ptr,
                                                 const uint32_t* __restrict__ col,
                                                 const uint32_t* __restrict__ off,
                                                 const uint32_t* __restrict__ defer,
                                                 const uint32_t* __restrict__ dcnt, uint32_t colour,
                                                 const double4_32a* __restrict__ prop,
                                                 uint8_t* __restrict__ acc,
                                                 DevCounters* __restrict__ cnt) {
  const uint32_t b = off[colour], n = dcnt[colour];
  const int lane = threadIdx.x & 31;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  unsigned ndd = 0;
  for (uint32_t q = warp; q < n; q += nwarps) {
    const uint32_t i = defer[b + q];
    const bool ok = settle_site(P, i, sw, s, row_ptr, col, prop, lane, ndd);
    if (lane == 0) {
      SiteCtx c;
      load_site(P, c, i, s);
      take_proposal(c, prop);
      write_site(P, c, ok, s, s32, acc);
    }
    __syncwarp();
  }
  if (lane == 0 && ndd) atomicAdd(&cnt->guard_fp64, (unsigned long long)ndd);
}

}  // namespace

cudaError_t sweep_run(const DevParams& P, const Table& t, double* s, float4* s32, SpinDf* sd,
                      const uint32_t* row_ptr, const uint32_t* col, const uint32_t* perm,
                      const uint32_t* off, uint32_t g, uint64_t step, int precision,
                      uint8_t* acc, uint32_t* defer, uint32_t* dcnt, double4_32a* prop,
                      SpinDf* propd, DevCounters* cnt, cudaStream_t st, int64_t* launches) {
  k_propose<<<(unsigned)((P.N + 255) / 256), 256, 0, st>>>(P, step, prop,
                                                           precision == 1 ? nullptr : propd);
  ++*launches;
  const unsigned grid = (unsigned)(8 * num_sms());  // the resident blocks of __launch_bounds__
  if (precision != 1) {
    const SweepArgs A{t.pdf, t.sw64, s, sd, row_ptr, col, perm, off, prop, propd, acc, cnt};
    for (uint32_t c = 0; c < g; ++c) {
      k_sweep_df<<<grid, 128, 0, st>>>(P, A, c);
      ++*launches;
    }
    return cudaGetLastError();
  }
  cudaError_t e = cudaMemsetAsync(dcnt, 0, (size_t)g * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  for (uint32_t c = 0; c < g; ++c) {
    k_sweep32<<<grid, 128, 0, st>>>(P, t.sw32, s, s32, row_ptr, col, perm, off, c, prop, acc,
                                    defer, dcnt, cnt);
    k_resolve<<<(unsigned)(4 * num_sms()), 128, 0, st>>>(P, t.sw64, s, s32, row_ptr, col, off,
                                                         defer, dcnt, c, prop, acc, cnt);
    *launches += 2;
  }
  return cudaGetLastError();
}

}  // namespace sco
