// switch.cu -- step (A) of Sec. 2.1 (potential switching) for one lattice and the
// compaction of the surviving pairs into a symmetric CSR graph.  The per-site body (bound
// thinning over the sorted half-plane list, exact decisions) is in switch_dev.cuh.
#include <algorithm>
#include <cstdint>

#include "switch_dev.cuh"

namespace sco {

namespace {

// Persistent: the warps claim the lattice's sites from a global counter (switch_range).
// Bound by instruction issue (58% busy, 24 of 32 lanes active) and the latency of the neighbours'
// records.  Four blocks per SM (64 registers; three and five measured 0.3 and 0.25 ms slower at
// L = 2304).  With the guided search, the float-float survival test and two candidates per step the
// FP64 form's switch phase takes 2.92 ms at L = 2304, T = 0.6 D (6.25 before), the FP32-screened
// one 2.60 (5.87).  Searching both candidates before testing either took 3.13 (spills), with
// prefetches of their records 3.74.
template <int PREC>
__global__ void __launch_bounds__(256, 4) k_switch(const __grid_constant__ DevParams P,
                                                   const __grid_constant__ Search S,
                                                   const SwitchIn in, uint32_t epoch, int32_t mnn0,
                                                   int32_t mnn1, SwitchBufs b,
                                                   DevCounters* __restrict__ cnt) {
  __shared__ NearShared sh;
  const NearTable T = near_table(S, sh);
  __syncthreads();
  const SwitchOut o{b.hslot, b.indeg, b.ovf, b.ovf_cap, &cnt->ovf_n, &cnt->ovf_full};
  unsigned n_dip = 0, ghits = 0, g32 = 0;
  const unsigned n_half =
      switch_range<PREC, true>(P, T, in, epoch, mnn0, mnn1, &cnt->sw_next, (uint32_t)P.N, 0u, b.hcnt, o,
                         n_dip, ghits, g32);
  const unsigned long long nh = warp_sum_u64(n_half), ndp = warp_sum_u64(n_dip);
  const unsigned long long gh = warp_sum_u64(ghits), gl = warp_sum_u64(g32);
  if ((threadIdx.x & 31) == 0) {
    if (nh) atomicAdd(&cnt->n_half, nh);
    if (ndp) atomicAdd(&cnt->n_dip, ndp);
    if (gh) atomicAdd(&cnt->guard_fp64, gh);
    if (gl) atomicAdd(&cnt->guard_fp32, gl);
  }
}

__global__ void k_degree(int64_t N, const uint32_t* __restrict__ hcnt,
                         const uint32_t* __restrict__ indeg, uint32_t* __restrict__ deg,
                         DevCounters* __restrict__ cnt) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned m = 0;
  if (i < N) {
    m = hcnt[i] + indeg[i];
    deg[i] = m;
  } else if (i == N) {
    deg[N] = 0;
  }
  // most warps stay at or below the running maximum: reading it first keeps their atomics off the
  // one address (113 us at L = 2304 with an atomic per warp)
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned*)&cnt->max_degree)
    atomicMax(&cnt->max_degree, m);
}

__global__ void k_fill(int64_t N, RowFill F, const uint32_t* __restrict__ hslot,
                       const uint32_t* __restrict__ hcnt, const uint32_t* __restrict__ indeg,
                       const uint32_t* __restrict__ row_ptr, uint32_t* __restrict__ cur,
                       uint32_t* __restrict__ col) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < N)
    fill_rows(F, (uint32_t)i, hslot + i * (int64_t)kSlotCap, hcnt[i], indeg, row_ptr, cur, col);
}

__global__ void k_fill_ovf(unsigned long long n, RowFill F, const uint32_t* __restrict__ ovf,
                           const uint32_t* __restrict__ row_ptr,
                           const uint32_t* __restrict__ indeg, uint32_t* hcnt,
                           uint32_t* __restrict__ cur, uint32_t* __restrict__ col) {
  const unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (q < n) fill_overflow(F, ovf[2 * q], ovf[2 * q + 1], row_ptr, indeg, hcnt, cur, col);
}

// Rows sorted by neighbour index (distinct inside a row) into `out`, a warp per row: an entry's place is
// the number of smaller ones, counted by shuffles of 32 entries at a time.  A thread per row took 0.50 ms
// of the getter's 0.80 at L = 256, T = 0.05 D (insertion from 32 entries on).
__global__ void __launch_bounds__(256) k_rowsort(int64_t N, const uint32_t* __restrict__ row_ptr,
                                                 uint32_t first, const uint32_t* __restrict__ col,
                                                 uint32_t* __restrict__ out,
                                                 DevCounters* __restrict__ cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  unsigned dmax = 0;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < N;
       i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const uint32_t b = row_ptr[i], n = row_ptr[i + 1] - b;
    const uint32_t* src = col + b;
    uint32_t* dst = out + (b - first);
    unsigned nd = 0;
    for (uint32_t a = 0; a < n; a += 32) {
      const bool on = a + lane < n;
      const uint32_t v = on ? src[a + lane] : kIndexMask, key = v & kIndexMask;
      uint32_t rank = 0;
      for (uint32_t c = 0; c < n; c += 32) {
        const uint32_t x = c + lane < n ? src[c + lane] & kIndexMask : kIndexMask;
        const uint32_t m = min(32u, n - c);
        for (uint32_t q = 0; q < m; q += 8) {
#pragma unroll
          for (uint32_t k = 0; k < 8; ++k) rank += __shfl_sync(0xffffffffu, x, q + k) < key ? 1u : 0u;
        }
      }
      if (on) dst[rank] = v;
      nd += (unsigned)__popc(__ballot_sync(0xffffffffu, on && !(v & kExchOnly)));
    }
    dmax = max(dmax, nd);
  }
  if (lane == 0 && dmax > *(volatile unsigned*)&cnt->max_degree_dip)
    atomicMax(&cnt->max_degree_dip, dmax);
}

}  // namespace

cudaError_t switch_run(const DevParams& P, const Table& t, const double* s, const float4* s32,
                       const SpinDf* sd, int precision, uint32_t epoch, SwitchBufs& b, DevCounters* cnt,
                       cudaStream_t st, int64_t* launches) {
  cudaError_t e = cudaMemsetAsync(b.indeg, 0, P.N * sizeof(uint32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(&cnt->sw_next, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  if (P.N <= 0) return cudaSuccess;
  // persistent grid: the resident blocks, at most one thread per site
  static int bps[2] = {0, 0};
  const int pi = precision == 1 ? 1 : 0;
  if (bps[pi] == 0) {
    e = pi ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps[pi], k_switch<1>, 256, 0)
           : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps[pi], k_switch<0>, 256, 0);
    if (e != cudaSuccess) return e;
    if (bps[pi] < 1) bps[pi] = 1;
  }
  int64_t nb64 = (int64_t)bps[pi] * num_sms();
  if (nb64 > (P.N + 255) / 256) nb64 = (P.N + 255) / 256;
  const unsigned nb = (unsigned)nb64;
  const Search S = table_search(t, t);
  const SwitchIn in{t.pdf, t.qdf, t.xy32, s, s32, sd};
  if (precision == 1)
    k_switch<1><<<nb, 256, 0, st>>>(P, S, in, epoch, t.m_nn[0], t.m_nn[1], b, cnt);
  else
    k_switch<0><<<nb, 256, 0, st>>>(P, S, in, epoch, t.m_nn[0], t.m_nn[1], b, cnt);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t csr_scan(const DevParams& P, SwitchBufs& b, uint32_t* row_ptr, DevCounters* cnt,
                     cudaStream_t st, int64_t* launches) {
  k_degree<<<(unsigned)((P.N + 1 + 255) / 256), 256, 0, st>>>(P.N, b.hcnt, b.indeg, b.deg, cnt);
  ++*launches;
  return scan_excl_u32(b.deg, row_ptr, P.N + 1, b.scan_tmp,
                       reinterpret_cast<uint64_t*>(&cnt->nnz), st, launches);
}

cudaError_t csr_fill(const DevParams& P, const SwitchBufs& b, uint32_t g, const uint32_t* row_ptr,
                     uint32_t* col, bool has_overflow, DevCounters* cnt, cudaStream_t st,
                     int64_t* launches) {
  cudaError_t e = cudaMemsetAsync(b.lcur, 0, P.N * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  const unsigned nb = (unsigned)((P.N + 255) / 256);
  const RowFill F = row_fill(g, (uint32_t)P.Lx, P.N, flow_max_pal(P.N));
  k_fill<<<nb, 256, 0, st>>>(P.N, F, b.hslot, b.hcnt, b.indeg, row_ptr, b.lcur, col);
  ++*launches;
  if (has_overflow) {
    unsigned long long n = 0;
    e = cudaMemcpyAsync(&n, &cnt->ovf_n, sizeof(n), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (n > b.ovf_cap) n = b.ovf_cap;
    if (n > 0) {
      k_fill_ovf<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, F, b.ovf, row_ptr, b.indeg, b.hcnt,
                                                                b.lcur, col);
      ++*launches;
    }
  }
  return cudaGetLastError();
}

cudaError_t csr_sorted_copy(const DevParams& P, const uint32_t* row_ptr, const uint32_t* col,
                            uint32_t first, uint64_t nnz, SortWork& w, DevCounters* cnt,
                            cudaStream_t st, int64_t* launches) {
  if (w.cap < nnz || !w.p) {
    w.release();
    const uint64_t cap = nnz <= kSortKeep ? nnz + nnz / 4 : nnz;
    const cudaError_t e = cudaMalloc(&w.p, cap * sizeof(uint32_t));
    if (e != cudaSuccess) {
      w.p = nullptr;
      return e;
    }
    w.cap = cap;
  }
  const int64_t nb = (P.N + 7) / 8;
  k_rowsort<<<(unsigned)std::min<int64_t>(nb, 64 * (int64_t)num_sms()), 256, 0, st>>>(
      P.N, row_ptr, first, col, w.p, cnt);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace sco
