// kw_static.cu -- Kuhn-Wattenhofer colouring of a caller's CSR graph that allocates nothing.
//
// Same colouring as sco_colour (palettes of at most 255 colours by the dataflow kernel of
// kw_flow.cuh, larger ones and sparse scattered graphs by one barrier-free kernel per level), for
// callers that cannot let a library allocate device memory.  Its working memory is one file-scope
// device array of fixed size: per-vertex words for up to SCO_KW_STATIC_MAX_VERTICES vertices followed
// by a small control block.  Every call shares that array; calls that overlap on the GPU race.
#include <cstdint>
#include <cstring>
#include <mutex>

#include "kw_flow.cuh"
#include "sco.h"
#include "sco_internal.h"

namespace sco {

namespace {

constexpr int64_t kMaxVertices = SCO_KW_STATIC_MAX_VERTICES;
constexpr int kCtrlWords = 64;  // 512 bytes of control block after the vertex words
constexpr int kMaxDevices = 64;

struct StaticCtrl {
  unsigned int max_degree;
  unsigned int g;
  unsigned int levels;
  int status;
  unsigned long long magic;  // multiplier of g (div_magic)
  unsigned int kw_rounds;
  unsigned int seen, far;    // sampled entries, and those that join distant vertices
  unsigned int entries;
  unsigned int lev_rounds[32];
  RepPlan plan;  // the dataflow kernel's view of the one lattice
  unsigned int site_start[2];
  unsigned int bar[2];
};
static_assert(sizeof(StaticCtrl) <= kCtrlWords * 8, "control block");

// The scratch: kMaxVertices packed words, then the control block.  8 MiB + 512 B per device.
static __device__ __align__(256) unsigned long long g_kw_scratch[kMaxVertices + kCtrlWords];

// The larger graphs' first entries of about 256 rows say whether neighbours lie near one another (see
// scattered_static).
constexpr uint32_t kScatterMin = 1u << 14, kSampledRows = 256, kSampledEntries = 4;

__global__ void k_st_degree(uint32_t n, const uint32_t* __restrict__ row_ptr,
                            const uint32_t* __restrict__ col, StaticCtrl* __restrict__ ctrl) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned d = v < n ? row_ptr[v + 1] - row_ptr[v] : 0u;
  if (v == 0) ctrl->entries = row_ptr[n] - row_ptr[0];
  if (n >= kScatterMin && d > 0 && v % (n / kSampledRows) == 0) {
    const uint32_t m = min(d, kSampledEntries), b = row_ptr[v];
    uint32_t u[kSampledEntries];
#pragma unroll
    for (uint32_t q = 0; q < kSampledEntries; ++q) u[q] = q < m ? col[b + q] & kIndexMask : v;
    unsigned far = 0;
#pragma unroll
    for (uint32_t q = 0; q < kSampledEntries; ++q)
      far += (u[q] > v ? u[q] - v : v - u[q]) > n / 64 ? 1u : 0u;
    atomicAdd(&ctrl->seen, m);
    if (far) atomicAdd(&ctrl->far, far);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d = max(d, __shfl_down_sync(0xffffffffu, d, o));
  if ((threadIdx.x & 31) == 0 && d) atomicMax(&ctrl->max_degree, d);
}

__global__ void k_st_setup(uint32_t n, StaticCtrl* __restrict__ ctrl) {
  const unsigned g = ctrl->max_degree + 1;
  const uint32_t G = (n + g - 1) / g;
  unsigned M = 0;
  while ((1u << M) < G) ++M;
  ctrl->g = g;
  ctrl->levels = M;
  ctrl->magic = div_magic(g);
  ctrl->plan = RepPlan{g, (uint16_t)M, 0, div_magic(g)};
  ctrl->site_start[0] = 0;
  ctrl->site_start[1] = n;
}

__global__ void k_st_init(uint32_t n, unsigned long long* __restrict__ word,
                          const StaticCtrl* __restrict__ ctrl) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) word[v] = pack(0, 0, v % ctrl->g);
}

__global__ void k_st_flow_init(uint32_t n, uint32_t g, uint32_t m32, uint32_t* __restrict__ word) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) word[v] = v - flow_div(v, g, m32) * g;
}

__device__ __noinline__ unsigned st_mex_slow(uint32_t v, unsigned p, unsigned long long M,
                                             const uint32_t* __restrict__ row_ptr,
                                             const uint32_t* __restrict__ col,
                                             const unsigned long long* word) {
  const uint32_t b = row_ptr[v], e = row_ptr[v + 1];
  const uint32_t grp = fdiv(v, M) >> p;
  for (unsigned c = 0;; ++c) {
    bool used = false;
    for (uint32_t q = b; q < e && !used; ++q) {
      const uint32_t u = col[q] & kIndexMask;
      const uint32_t gu = fdiv(u, M);
      if ((gu >> p) != grp) continue;
      const unsigned long long wu = ld_relaxed(&word[u]);
      if (((gu >> (p - 1)) & 1u) && tag_of(wu) != p) continue;
      used = (unsigned)(wu & kColMask) == c;
    }
    if (!used) return c;
  }
}

// Sparse graphs whose neighbours lie anywhere are coloured level by level as well: hardly a vertex finds
// its neighbours in its block then, the chains are short, and the dataflow kernel's sort and barrier per
// level are not repaid.  Neighbours further apart than n / 64 make up most of the sampled entries.  Dataflow
// kernel and level kernels, in us: a shuffled path, n = 30,000 161 and 156, 100,000 190 and 174, 1,000,000
// 514 and 349 (in order 477 and 521); a shuffled square grid, n = 100,000 189 and 205, 200,000 241 and 218,
// 1,000,000 536 and 404 (in order 526 and 759); six random matchings, n = 1,000,000 551 and 466; its
// 8-neighbour grid, shuffled, 554 and 561; random graphs of mean degree 1 and 2, n = 200,000 221 and 196,
// 221 and 220; 3 and 4, n = 400,000 280 and 268, 281 and 287; 5 and 6, n = 1,000,000 513 and 497, 529 and 550.
inline bool scattered_static(const StaticCtrl& c, uint32_t n) {
  if (n < kScatterMin || c.seen == 0 || 2 * c.far <= c.seen) return false;
  return c.g <= 3 || (n >= (1u << 17) && (c.g <= 7 || c.entries < (double)n * n / 187000.0));
}

// One KW level (modified reduction (2)') of a graph that the dataflow kernel does not take; g, M and
// the divisor constant come from the control block.
__global__ void __launch_bounds__(256) k_st_level(uint32_t n, unsigned p,
                                                  const uint32_t* __restrict__ row_ptr,
                                                  const uint32_t* __restrict__ col,
                                                  unsigned long long* word,
                                                  StaticCtrl* __restrict__ ctrl,
                                                  unsigned long long ns_limit) {
  if (p > ctrl->levels) return;
  const unsigned long long t_start = global_ns();
  const uint32_t g = ctrl->g;
  const unsigned long long M = ctrl->magic;
  const uint32_t half = g << (p - 1);
  const uint32_t ngroups = (uint32_t)(((unsigned long long)n + ((unsigned long long)g << p) - 1) /
                                      ((unsigned long long)g << p));
  const uint32_t R = ngroups * half;
  const uint32_t nth = gridDim.x * blockDim.x;
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned rmax = 0;
  unsigned nap = 64;  // back-off (ns) after a pass in which none of this thread's vertices moved
  bool pending = true;
  for (unsigned long long pass = 0; pending; ++pass) {
    pending = false;
    bool progress = false;
    for (uint32_t r = tid; r < R; r += nth) {
      const uint32_t k = fdiv(r, M) >> (p - 1);
      const uint32_t v = (2 * k + 1) * half + (r - k * half);
      if (v >= n) continue;
      const unsigned long long wv = ld_relaxed(&word[v]);
      if (tag_of(wv) == p) continue;
      const uint32_t cv = (uint32_t)(wv & kColMask);
      const uint32_t b = row_ptr[v], e = row_ptr[v + 1];
      unsigned long long used[4] = {0, 0, 0, 0};
      bool blocked = false;
      unsigned rv = 0;
      for (uint32_t q = b; q < e; ++q) {
        const uint32_t u = col[q] & kIndexMask;
        const uint32_t gu = fdiv(u, M);
        if ((gu >> p) != k) continue;
        const unsigned long long wu = ld_relaxed(&word[u]);
        const uint32_t cu = (uint32_t)(wu & kColMask);
        const bool right = (gu >> (p - 1)) & 1u;
        if (right && tag_of(wu) != p) {
          if (cu > cv) {
            blocked = true;
            break;
          }
          continue;
        }
        if (right) rv = max(rv, rnd_of(wu));
        if (cu < 256) used[cu >> 6] |= 1ull << (cu & 63);
      }
      if (blocked) {
        pending = true;
        continue;
      }
      unsigned c = 0;
      if (e - b < 256) {
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          if (~used[w]) {
            c = 64 * w + __ffsll((long long)~used[w]) - 1;
            break;
          }
        }
      } else {
        c = st_mex_slow(v, p, M, row_ptr, col, word);
      }
      rmax = max(rmax, rv + 1);
      st_relaxed(&word[v], pack(p, rv + 1, c));
      progress = true;
    }
    if (pending) {
      if (progress) {
        nap = 64;
      } else {
        __nanosleep(nap);
        nap = nap < 2048 ? 2 * nap : 2048;
      }
    }
    if (pending && ((pass & 15) == 15) &&
        (global_ns() - t_start > ns_limit || ld_status(&ctrl->status) != 0)) {
      atomicCAS(&ctrl->status, 0, kStatusTimeout);
      break;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rmax = max(rmax, __shfl_down_sync(0xffffffffu, rmax, o));
  if ((threadIdx.x & 31) == 0 && rmax) atomicMax(&ctrl->lev_rounds[p & 31], rmax);
}

// fword: the dataflow kernel's words (null: word)
__global__ void k_st_final(uint32_t n, int variant, const unsigned long long* __restrict__ word,
                           const uint32_t* __restrict__ fword, uint32_t* __restrict__ colour,
                           StaticCtrl* __restrict__ ctrl) {
  const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) colour[v] = fword ? fword[v] & 0xFFu : (uint32_t)(word[v] & kColMask);
  if (v == 0) {
    unsigned t = 0;
    for (unsigned p = 1; p <= ctrl->levels; ++p) t += ctrl->lev_rounds[p & 31];
    ctrl->kw_rounds = variant == 1 ? ctrl->g * ctrl->levels : t;
  }
}

std::mutex g_setup_mu;
unsigned long long* g_scratch_addr[kMaxDevices] = {};
int g_blocks_per_sm[kMaxDevices] = {};
int g_sms[kMaxDevices] = {};

}  // namespace

}  // namespace sco

using namespace sco;

extern "C" sco_status sco_kw_colour_static(const uint32_t* row_ptr, const uint32_t* col,
                                           int64_t n, int32_t variant, uint32_t* colour,
                                           int32_t* max_degree, int32_t* rounds, void* stream) {
  if (n < 0 || n > kMaxVertices || variant < 0 || variant > 1) return SCO_EINVAL;
  if (n == 0) {
    if (max_degree) *max_degree = 0;
    if (rounds) *rounds = 0;
    return SCO_OK;
  }
  if (!row_ptr || !col || !colour) return SCO_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SCO_ECUDA;
  unsigned long long* base = nullptr;
  {
    // once per device, with that device current: the device address of the scratch array
    std::lock_guard<std::mutex> lock(g_setup_mu);
    if (!g_scratch_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_kw_scratch) != cudaSuccess || !p) return SCO_ECUDA;
      int bps = 0, sms = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_st_level, 256, 0) != cudaSuccess)
        return SCO_ECUDA;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return SCO_ECUDA;
      g_blocks_per_sm[dev] = bps > 0 ? bps : 1;
      g_sms[dev] = sms > 0 ? sms : 1;
      g_scratch_addr[dev] = (unsigned long long*)p;
    }
    base = g_scratch_addr[dev];
  }
  unsigned long long* word = base;
  StaticCtrl* ctrl = reinterpret_cast<StaticCtrl*>(base + kMaxVertices);
  const uint32_t nn = (uint32_t)n;
  if (cudaMemsetAsync(ctrl, 0, sizeof(StaticCtrl), st) != cudaSuccess) return SCO_ECUDA;
  const unsigned nb = (nn + 255) / 256;
  k_st_degree<<<nb, 256, 0, st>>>(nn, row_ptr, col, ctrl);
  k_st_setup<<<1, 1, 0, st>>>(nn, ctrl);
  // Delta and the sample decide the kernel: small palettes mostly run the dataflow kernel
  StaticCtrl h;
  std::memset(&h, 0, sizeof(h));
  if (cudaMemcpyAsync(&h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return SCO_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return SCO_ECUDA;
  unsigned long long ns_limit = 2000000000ull;
  FlowShape shape;
  cudaError_t fe = cudaSuccess;
  const bool flow = h.g <= kFlowMaxPal && h.levels < kFlowMaxLevels && !scattered_static(h, nn) &&
                    flow_shape(1, nn, h.g, &shape, &fe);
  if (fe != cudaSuccess) return SCO_ECUDA;
  uint32_t* fword = flow ? reinterpret_cast<uint32_t*>(word) : nullptr;
  if (flow) {
    k_st_flow_init<<<nb, 256, 0, st>>>(
        nn, h.g, h.g > 1 ? (uint32_t)(0x100000000ull / h.g) : 0xFFFFFFFFu, fword);
    FlowView F{};
    F.R = 1;
    F.site_start = ctrl->site_start;
    F.plan = &ctrl->plan;
    F.row_ptr = row_ptr;
    F.col = col;
    F.word = fword;
    F.lev_rounds = ctrl->lev_rounds;
    F.bar = ctrl->bar;
    F.status = &ctrl->status;
    F.levels = h.levels;
    F.cap = shape.cap;
    F.min_tile = shape.min_tile;
    F.ns_limit = ns_limit;
    F.vec = ((uintptr_t)col & 31u) == 0 ? kFlowVecInside : kFlowVecNone;
    if (flow_launch(F, shape, st) != cudaSuccess) return SCO_ECUDA;
  } else {
    k_st_init<<<nb, 256, 0, st>>>(nn, word, ctrl);
    if (cudaGetLastError() != cudaSuccess) return SCO_ECUDA;
    int64_t grid = (int64_t)g_blocks_per_sm[dev] * g_sms[dev];
    const int64_t want = ((int64_t)nn / 2 + 255) / 256;
    if (want < grid) grid = want > 0 ? want : 1;
    for (unsigned p = 1; p <= h.levels; ++p) {
      uint32_t a0 = nn;
      unsigned a1 = p;
      void* args[] = {(void*)&a0, (void*)&a1, (void*)&row_ptr, (void*)&col, (void*)&word,
                      (void*)&ctrl, (void*)&ns_limit};
      if (cudaLaunchCooperativeKernel((const void*)k_st_level, dim3((unsigned)grid), dim3(256),
                                      args, 0, st) != cudaSuccess)
        return SCO_ECUDA;
    }
  }
  k_st_final<<<nb, 256, 0, st>>>(nn, variant, word, fword, colour, ctrl);
  if (cudaMemcpyAsync(&h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return SCO_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return SCO_ECUDA;
  if (h.status != 0) return (sco_status)h.status;
  if (max_degree) *max_degree = (int32_t)h.max_degree;
  if (rounds) *rounds = (int32_t)h.kw_rounds;
  return SCO_OK;
}
