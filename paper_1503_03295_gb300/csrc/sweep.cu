// sweep.cu -- step (B) of Sec. 2.1 / step (3) of Fig. 1 for one lattice: Metropolis
// updates of all sites of one colour class at a time.  Sites of one colour share no pair, so they
// update independently.  The per-site decisions and the kernel are in sweep_dev.cuh.
#include <algorithm>
#include <cstdint>

#include "sweep_dev.cuh"

namespace sco {

namespace {

// In the order of perm (see take_proposal).
__global__ void __launch_bounds__(256) k_propose(const DevParams P, uint64_t step,
                                                 const uint32_t* __restrict__ perm,
                                                 double4_32a* __restrict__ prop,
                                                 SpinDf* __restrict__ propd,
                                                 float4* __restrict__ prop32) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  write_proposal(P, step, perm[i], prop + i, propd ? propd + i : nullptr,
                 prop32 ? prop32 + i : nullptr);
}

}  // namespace

cudaError_t sweep_run(const DevParams& P, const Table& t, const SweepBufs& b, uint32_t g,
                      uint64_t step, int precision, DevCounters* cnt, unsigned long long ns_limit,
                      cudaStream_t st, int64_t* launches) {
  k_propose<<<(unsigned)((P.N + 255) / 256), 256, 0, st>>>(P, step, b.perm, b.prop, b.propd,
                                                             b.prop32);
  const int per = sweep_blocks(P.N, precision);
  const int64_t want = P.N <= kSweepOne ? 1 : (P.N + kSweepSites - 1) / kSweepSites;
  const unsigned grid = (unsigned)std::min<int64_t>(per * num_sms(), want);
  SweepView V{};
  V.R = 1;
  V.P = P;
  V.pdf = t.pdf;
  V.sw32 = t.sw32;
  V.sw = t.sw64;
  V.s = b.s;
  V.s32 = b.s32;
  V.sd = b.sd;
  V.row_ptr = b.row_ptr;
  V.col = b.col;
  V.perm = b.perm;
  V.off = b.off;
  V.prop = b.prop;
  V.propd = b.propd;
  V.prop32 = b.prop32;
  V.acc = b.acc;
  V.cnt = cnt;
  V.g = g;
  V.bar = cnt->bar;
  V.status = &cnt->status;
  V.ns_limit = ns_limit;
  void* args[] = {(void*)&V};
  *launches += 2;
  const void* k = P.J != 0.0 ? sweep_kernel<false, true>(precision, per)
                              : sweep_kernel<false, false>(precision, per);
  if (grid == 1) return cudaLaunchKernel(k, dim3(1), dim3(kSweepThreads), args, sweep_smem(1), st);
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kSweepThreads), args, sweep_smem(1), st);
}

}  // namespace sco
