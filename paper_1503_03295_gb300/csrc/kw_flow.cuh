// kw_flow.cuh -- all levels of the Kuhn-Wattenhofer colouring (Sec. 2.3.3) in one persistent
// cooperative kernel, by dataflow: a right-half vertex recolours as soon as its same-group
// right-half neighbours of larger previous colour have done so (modified reduction (2)' of
// Sec. 2.3.2; its colour and round do not depend on the order, see colour.cu).
//
// What bounds a level is the chain of dependent recolourings (about Delta + 1 long) and, for large
// lattices, the pass over the rows of the right-half vertices (instruction issue).  So a block owns
// a contiguous range of the level's right-half slots and keeps their words in shared memory: a hop
// of the chain between two vertices of one block costs a few hundred cycles, not a grid barrier
// (2 us) or a trip through L2 (1 to 2 us).  A range of a few lattice rows holds most of a vertex's
// right-half neighbours (about 72% for 7.6 rows at L = 2304); the others are read in global memory,
// where every recoloured vertex publishes its word.
//
// Inside a block the vertices are sorted by previous colour, largest first, and dealt to the warps
// 32 at a time in that order.  A lane reads its vertex's row once, adds what is final to the
// vertex's colour set and lists the larger neighbours that are not done; then the warp polls the
// lists until every lane has recoloured: nothing waits for a barrier, and a step of the chain is
// one poll of a short list.  No cycle of waits can form: a vertex only waits for larger previous
// colours, every warp takes its vertices in descending order, and all blocks are resident
// (cooperative launch).  Palettes of at most 255 colours; one lattice or a batch of them.
//
// Per colouring, by rounds and buckets (kw_low.cuh, kw_bcr.cuh, k_kw_level) and here: L = 2304, T =
// 0.6 D 6.63 -> 3.60 ms, L = 1024, T = 0.4 D 3.47 -> 1.10, 1000 x 1337, T = 0.8 D 2.57 -> 0.92, L =
// 256 1.74 -> 0.34, a static graph of 400,000 vertices 2.47 -> 0.44.  At L = 1500 it issues on 58% of
// the cycles with 22 of 32 lanes active, the ALU pipe 53% busy, DRAM 9%; the waits are for rows and
// words in L2 (4.0 warps per issue) and at the ends of the levels (2.3).
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "batch.h"
#include "grid_dev.cuh"
#include "kw_dev.cuh"

namespace sco {
namespace {

constexpr uint32_t kFlowKeys = 256;  // sort keys (flow_key)
constexpr unsigned kFlowMaxLevels = 32;
// Per lane: list entries (a longer row is read in parts; 40 in place of 24 took L = 1024, T = 0.4 D,
// mean degree 23, from 1.36 to 1.23 ms per colouring, but does not fit beside the words of a large
// lattice's blocks), and neighbours outside the block looked up together.
__host__ __device__ constexpr int flow_list(int threads) { return threads == 512 ? 40 : 24; }
__host__ __device__ constexpr int flow_look(int threads) { return threads == 512 ? 8 : 6; }
constexpr int kFlowChunk = 8;          // row entries read together (a multiple of 8)

struct FlowView {
  int R;                       // lattices (1 for a single lattice)
  const uint32_t* site_start;  // R + 1 first vertex of each lattice
  const RepPlan* plan;         // R: g, levels, near, magic
  const uint32_t* row_ptr;     // global entry offsets; col entries lattice-local
  const uint32_t* col;
  const uint32_t* rows;        // near entries of a row in the high half (see RowFill; null: no plan has near)
  // global vertex index: level << 27 | round << 8 | colour, the level and round of the last
  // recolouring; level 0 and the initial colour on entry
  uint32_t* word;
  unsigned* lev_rounds;        // lattice r's deepest round per level: lev_rounds + r * lev_stride
  uint32_t lev_stride;
  unsigned* bar;               // grid barrier words
  int* status;                 // sticky error word
  const int* halt;             // optional: nonzero on entry -> return at once
  const unsigned* gmax;        // optional: largest palette, on the device; above kFlowMaxPal -> return
  unsigned levels;             // >= every M, < kFlowMaxLevels
  uint32_t cap;                // right-half vertices a block holds, < 65535
  uint32_t min_tile;           // and at least owns (fewer blocks work on a small level)
  unsigned long long ns_limit;
  int vec;                     // kFlowVec*: which row entries may be read by whole sectors
};
// none (col not 32-byte aligned), those of whole sectors before the last entry of lattice 0 (a
// caller's array), or all (col is readable to a multiple of 8 entries)
constexpr int kFlowVecNone = 0, kFlowVecInside = 1, kFlowVecAll = 2;


// Dynamic shared memory: sites and slots per lattice (R + 1 each), rounds (R), sort cursors; a word
// and an order entry per owned vertex; the lanes' lists.
inline size_t kw_flow_smem(int R, uint32_t cap, int threads) {
  return (size_t)(3 * R + 2 + kFlowKeys) * sizeof(uint32_t) + (size_t)cap * 6 + 32 +
         (size_t)threads * flow_list(threads) * sizeof(uint16_t);
}

__device__ __forceinline__ uint32_t flow_ld(const uint32_t* p) { return ld_u32_gpu(p); }
__device__ __forceinline__ uint32_t flow_ld_if(const uint32_t* p, uint32_t on) {
  uint32_t v = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.relaxed.gpu.global.u32 %0, [%1];\n\t}"
      : "+r"(v)
      : "l"(p), "r"(on)
      : "memory");
  return v;
}
__device__ __forceinline__ void flow_st(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Right-half slots of a lattice of N vertices at level p that hold a vertex (the last group may be
// short): slot s of group k is vertex s + (k + 1) half.
__device__ __forceinline__ uint32_t flow_slots(uint32_t N, uint32_t g, unsigned p) {
  const unsigned long long gsz = (unsigned long long)g << p, half = gsz >> 1;
  const unsigned long long full = N / gsz, rem = N - full * gsz;
  return (uint32_t)(full * half + (rem > half ? rem - half : 0ull));
}

// u / g: one 32-bit multiply, corrected (see site_xy)
__device__ __forceinline__ uint32_t flow_div(uint32_t u, uint32_t g, uint32_t m32) {
  uint32_t q = __umulhi(u, m32);
  if (u - q * g >= g) ++q;
  return q;
}
__device__ __forceinline__ uint32_t flow_magic(uint32_t g) {
  return g > 1 ? (uint32_t)(0x100000000ull / g) : 0xFFFFFFFFu;
}

// Sort key of a vertex: previous colour, largest first, then (palettes up to 64) the number of
// eight-entry sectors of its row, so that the lanes of a warp read about the same number of them;
// kFlowKeys: no vertex.
__device__ __forceinline__ uint32_t flow_key(uint32_t c, uint32_t b, uint32_t e, uint32_t pal) {
  const uint32_t ns = ((e + 7) >> 3) - (b >> 3);
  return pal > 64 ? 255u - c : 4 * (63u - c) + (ns < 3 ? 0u : min(ns - 2, 3u));
}
// Word of a vertex in shared memory: round << 8 | colour once it is done, before that 2^31 | previous
// colour << 16 | kFlowNone.  A done right-half neighbour is a larger one (a smaller one waits for
// this vertex), so only open ones are compared.  flow_bit(kFlowNone) is no colour.
constexpr uint32_t kFlowNone = 255u;

// 1 << c for c < 32, else 0 (shl clamps)
__device__ __forceinline__ uint32_t flow_bit(uint32_t c) {
  uint32_t b;
  asm("shl.b32 %0, 1, %1;" : "=r"(b) : "r"(c));
  return b;
}

__device__ __forceinline__ uint32_t flow_lds(const uint32_t* p) {
  return *reinterpret_cast<const volatile uint32_t*>(p);
}

template <int kT, int kOwn>
__global__ void __launch_bounds__(kT, 1) k_kw_flow(const __grid_constant__ FlowView V) {
  __shared__ int s_halt;
  if (threadIdx.x == 0)
    s_halt = (V.halt && ld_status(V.halt)) || ld_status(V.status) ||
             (V.gmax && *V.gmax > kFlowMaxPal);
  __syncthreads();
  if (s_halt) return;
  constexpr uint32_t T = kT, kFlowList = flow_list(kT), kFlowLook = flow_look(kT);
  extern __shared__ uint32_t fsm[];
  const int R = V.R;
  uint32_t* sbase = fsm;              // R + 1
  uint32_t* rp = sbase + R + 1;       // R + 1 slot prefix at this level
  uint32_t* smax = rp + R + 1;        // R deepest round in this block
  uint32_t* cur = smax + R;           // kFlowKeys counts, then cursors
  uint32_t* st = cur + kFlowKeys;     // cap words, and one that stays kFlowNone
  uint16_t* ord = reinterpret_cast<uint16_t*>(st + V.cap + 1);  // cap
  // this lane's list, entries 32 apart
  uint16_t* list = ord + V.cap + (threadIdx.x & ~31u) * kFlowList + (threadIdx.x & 31u);
  const uint32_t tid = threadIdx.x;
  const int lane = (int)(tid & 31);
  for (int r = tid; r <= R; r += T) sbase[r] = V.site_start[r];
  if (tid == 0) st[V.cap] = kFlowNone;
  const RepPlan pl0 = V.plan[0];
  const uint32_t vec_end = V.vec == kFlowVecAll      ? 0xFFFFFFFFu
                           : V.vec == kFlowVecInside ? V.row_ptr[V.site_start[1]]
                                                     : 0u;
  const uint32_t m0 = flow_magic(pl0.g);
  const uint32_t pal = V.gmax ? *V.gmax : pl0.g;
  bool ok = true;
  for (unsigned p = 1; p <= V.levels && ok; ++p) {
    __syncthreads();
    for (int r = tid; r < R; r += T) {
      const RepPlan pl = R == 1 ? pl0 : V.plan[r];
      rp[r] = p <= pl.levels ? flow_slots(sbase[r + 1] - sbase[r], pl.g, p) : 0u;
      smax[r] = 0;
    }
    if (tid < kFlowKeys) cur[tid] = 0;
    __syncthreads();
    if (tid < 32) {  // exclusive prefix, 32 lattices at a time
      uint32_t run = 0;
      for (int r0 = 0; r0 < R; r0 += 32) {
        const int r = r0 + lane;
        const uint32_t v = r < R ? rp[r] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += t;
        }
        if (r < R) rp[r] = run + x - v;
        run += __shfl_sync(0xffffffffu, x, 31);
      }
      if (lane == 0) rp[R] = run;
    }
    __syncthreads();
    const uint32_t total = rp[R];
    if (total == 0) continue;  // the same in every block: no lattice has this level (nor a later one)
    // this block's slots [s0, s0 + n): an equal share, at least min_tile, and for one lattice whole
    // groups where that costs at most a quarter more
    uint32_t own = max((total + gridDim.x - 1) / gridDim.x, V.min_tile);
    if (R == 1) {
      const uint32_t half = pl0.g << (p - 1);
      const unsigned long long up = (unsigned long long)((own + half - 1) / half) * half;
      if (up <= V.cap && up * 4 <= (unsigned long long)own * 5) own = (uint32_t)up;
    }
    own = min(own, V.cap);
    const uint32_t s0 = min(total, blockIdx.x * own), n = min(own, total - s0);
    // first entry of vertex gv's row that the level looks at (near_levels)
    auto row_begin = [&](uint32_t gv, int r) {
      const uint32_t near = R == 1 ? pl0.near : V.plan[r].near;
      return p <= near ? V.row_ptr[gv + 1] - (V.rows[gv] >> 16) : V.row_ptr[gv];
    };
    // lattice, group and offsets of a slot
    auto locate = [&](uint32_t slot, int& r, uint32_t& k, uint32_t& half) {
      r = R == 1 ? 0 : find_le(rp, R, slot);
      const uint32_t g = R == 1 ? pl0.g : V.plan[r].g;
      half = g << (p - 1);
      k = flow_div(slot - rp[r], g, R == 1 ? m0 : flow_magic(g)) >> (p - 1);
    };
    // the vertices per key, four loads of each array in flight
    for (uint32_t q0 = 0; q0 < n; q0 += 4 * T) {
      uint32_t c[4], rb[4], re[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const uint32_t q = q0 + a * T + tid;
        c[a] = rb[a] = re[a] = 0;
        if (q < n) {
          int r;
          uint32_t k, half;
          locate(s0 + q, r, k, half);
          const uint32_t gv = sbase[r] + (s0 + q - rp[r]) + (k + 1) * half;
          c[a] = flow_ld(&V.word[gv]);
          rb[a] = row_begin(gv, r);
          re[a] = V.row_ptr[gv + 1];
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const uint32_t q = q0 + a * T + tid;
        const uint32_t key = q < n ? flow_key(c[a] & 0xFFu, rb[a], re[a], pal) : kFlowKeys;
        if (q < n) st[q] = 0x80000000u | ((c[a] & 0xFFu) << 16) | (key << 8) | kFlowNone;
        if (q0 + a * T >= n) break;  // uniform
        if (q < n) atomicAdd(&cur[key], 1u);
      }
    }
    __syncthreads();
    if (tid < 32) {  // cur[key]: vertices of smaller keys
      uint32_t v[8], x = 0;
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        v[a] = cur[8 * lane + a];
        x += v[a];
      }
      const uint32_t mine = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
      }
      x -= mine;
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        cur[8 * lane + a] = x;
        x += v[a];
      }
    }
    __syncthreads();
    for (uint32_t q0 = 0; q0 < n; q0 += T) {
      const uint32_t q = q0 + tid;
      const uint32_t w = q < n ? st[q] : 0u;
      const uint32_t key = q < n ? (w >> 8) & 0xFFu : kFlowKeys;
      if (q < n) {
        ord[atomicAdd(&cur[key], 1u)] = (uint16_t)q;
        st[q] = w & 0xFFFF00FFu;
      }
    }
    __syncthreads();
    const unsigned long long t_start = global_ns();
    unsigned rmax = 0, spins = 0;
    for (uint32_t t0 = (tid & ~31u); t0 < n && ok; t0 += T) {
      bool open = t0 + lane < n;
      uint32_t loc = 0, c = 0, gv = 0, base = 0, lo = 0, half = 0, b = 0, e = 0;
      uint32_t fa = 0, len = 0, la = 0;
      uint32_t mlo = 0;  // colours below 32 taken
      int m = 0;         // the largest round << 8 (and bits below)
      int r = 0;
      auto add = [&](uint32_t w) { mlo |= flow_bit(w & 0xFFu); };
      if (open) {
        loc = ord[t0 + lane];
        uint32_t k;
        locate(s0 + loc, r, k, half);
        base = sbase[r];
        gv = base + (s0 + loc - rp[r]) + (k + 1) * half;
        b = row_begin(gv, r);
        e = V.row_ptr[gv + 1];
        c = (st[loc] >> 16) & 0xFFu;
        lo = 2 * k * half;
        // the block's part of the right half: vertices [fa, fa + len), words from la on
        const uint32_t h0 = k * half + rp[r], g0 = max(h0, s0), g1 = min(h0 + half, s0 + n);
        fa = g0 - rp[r] + (k + 1) * half;
        len = g1 - g0;
        la = g0 - s0;
      }
      const uint32_t lthr = 0x80000000u | (c << 16) | 0xFFFFu;  // open and larger: words above it
      const uint32_t done_at = p << 27;                           // done: global words from it on
      const uint32_t* own = st + la;
      const uint32_t none = V.cap - la;  // word cap: no colour
      uint32_t cnt = 0, fcnt = 0;        // listed: open vertices of this block, entries to look up
      uint32_t k = 0, f = 0;             // and how many of them are settled
      uint32_t q0 = b & ~7u;             // next sector of the row
      // recolours the lane's vertex: all its larger neighbours are done
      auto finish = [&]() {
        uint32_t cn = (uint32_t)__ffs((int)~mlo) - 1;
        for (uint32_t taken = mlo, c0 = 32; taken == 0xFFFFFFFFu; c0 += 32) {
          // rare: colours c0 .. c0 + 31, from the row again
          taken = 0;
          for (uint32_t q = b; q < e; ++q) {
            const uint32_t u = V.col[q] & kIndexMask;
            if (u - lo >= 2 * half) continue;
            const bool mine = u - fa < len, left = u - lo < half;
            const uint32_t y = mine ? flow_lds(own + (u - fa)) : flow_ld(&V.word[base + u]);
            if (left || (mine ? (int)y >= 0 : y >= done_at)) taken |= flow_bit((y & 0xFFu) - c0);
          }
          cn = c0 - 1 + (uint32_t)__ffs((int)~taken);
        }
        const uint32_t rd = (uint32_t)(m >> 8) + 1;
        *reinterpret_cast<volatile uint32_t*>(st + loc) = (rd << 8) | cn;
        flow_st(&V.word[gv], (p << 27) | (rd << 8) | cn);
        if (R == 1) rmax = max(rmax, rd);
        else atomicMax(&smax[r], rd);
        open = false;
      };
      // nothing moved for a while: true once a bounded wait gave up
      auto give_up = [&]() {
        const bool out = (++spins & wait_spin_mask(V.ns_limit)) == 0 &&
                         (global_ns() - t_start > V.ns_limit || ld_status(V.status) != 0);
        if (!__any_sync(0xffffffffu, out)) return false;
        if (lane == 0) atomicCAS(V.status, 0, kStatusTimeout);
        ok = false;
        return true;
      };
      while (__any_sync(0xffffffffu, open)) {
        if (!__any_sync(0xffffffffu, open && (q0 < e || f < fcnt))) {
          // only the block's own neighbours are left: a short loop, as its length is that of a hop of
          // the chain (L = 256 351 -> 338 us per colouring, 1024 FP32 1.13 -> 1.09 ms, L = 16 80 -> 76 us)
          do {
            uint32_t w[kOwn];
#pragma unroll
            for (int a = 0; a < kOwn; ++a)
              w[a] = flow_lds(own + (k + a < cnt ? (uint32_t)list[32 * (k + a)] : none));
            bool moved = false;
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
              if (k < cnt && (int)w[a] >= 0 && (a == 0 || moved)) {
                add(w[a]);
                m = max(m, (int)w[a]);
                ++k;
                moved = true;
              } else {
                break;
              }
            }
            if (open && k == cnt) {
              finish();
              moved = true;
            }
            if (!__any_sync(0xffffffffu, moved) && give_up()) break;
          } while (__any_sync(0xffffffffu, open));
          break;
        }
        bool moved = false;
        if (q0 < e && k == cnt && f == fcnt) {
          moved = true;
          cnt = fcnt = k = f = 0;
          // while a whole chunk fits the list
          for (; q0 < e && cnt + fcnt <= kFlowList - kFlowChunk; q0 += kFlowChunk) {
            uint32_t uu[kFlowChunk], w[kFlowChunk];
            // entries of [b, e) among the chunk's
            uint32_t in = e - q0 < kFlowChunk ? (1u << (e - q0)) - 1u : (1u << kFlowChunk) - 1u;
            if (q0 < b) in &= ~((1u << (b - q0)) - 1u);
            // whole sectors: a load of 32 rows takes 32 passes through L1 at any width
            if (q0 + kFlowChunk <= vec_end) {
#pragma unroll
              for (int a = 0; a < kFlowChunk; a += 8) {
                struct __align__(32) Eight { uint32_t v[8]; } t = {};
                if (q0 + a < e) t = load32(reinterpret_cast<const Eight*>(V.col + q0 + a));
#pragma unroll
                for (int h = 0; h < 8; ++h) uu[a + h] = t.v[h];
              }
            } else {
#pragma unroll
              for (int a = 0; a < kFlowChunk; ++a) uu[a] = (in >> a) & 1u ? V.col[q0 + a] : 0u;
            }
#pragma unroll
            for (int a = 0; a < kFlowChunk; ++a) {
              uu[a] &= kIndexMask;
              const bool on = ((in >> a) & 1u) && uu[a] - lo < 2 * half;  // in the group
              uu[a] -= fa;
              const bool mine = on && uu[a] < len;
              w[a] = flow_lds(own + (mine ? uu[a] : none));
              // the left half or another block's: its entry number
              if (on && !mine) list[32 * (kFlowList - 1 - fcnt++)] = (uint16_t)(q0 + a - b);
            }
#pragma unroll
            for (int a = 0; a < kFlowChunk; ++a) {
              if (w[a] > lthr) list[32 * cnt++] = (uint16_t)uu[a];
              add(w[a]);
              m = max(m, (int)w[a]);
            }
          }
        }
        // the lists in order, a few at a time, up to the first that is not done: the block's own beside
        // the looked-up ones, which wait for L2 (one list after the other, own ones four at a time:
        // L = 256 378 -> 351 us per colouring, 1000 x 1337 986 -> 933, L = 2304 3.68 -> 3.61 ms; own
        // ones by one 389 us, 934 us and 3.62 ms one after the other, by three 359, 951 and 3.63
        // beside)
        if (f < fcnt) {
          uint32_t u[kFlowLook], w[kFlowLook];
#pragma unroll
          for (uint32_t a = 0; a < kFlowLook; ++a)
            u[a] = f + a < fcnt ? V.col[b + list[32 * (kFlowList - 1 - f - a)]] & kIndexMask : kNone;
#pragma unroll
          for (uint32_t a = 0; a < kFlowLook; ++a) w[a] = flow_ld_if(&V.word[base + u[a]], f + a < fcnt);
          bool go = true;
#pragma unroll
          for (uint32_t a = 0; a < kFlowLook; ++a) {
            const uint32_t y = w[a];
            const bool left = u[a] - lo < half, done = y >= done_at;
            go = go && f < fcnt && (left || done || (y & 0xFFu) <= c);
            if (go) {
              if (left || done) add(y);
              if (!left && done) m = max(m, (int)(y & 0x7FFFFFFu));
              ++f;
              moved = true;
            }
          }
        }
        if (k < cnt) {
          uint32_t w[kOwn];
#pragma unroll
          for (int a = 0; a < kOwn; ++a)
            w[a] = flow_lds(own + (k + a < cnt ? (uint32_t)list[32 * (k + a)] : none));
          bool go = true;
#pragma unroll
          for (int a = 0; a < kOwn; ++a) {
            go = go && k < cnt && (int)w[a] >= 0;
            if (go) {
              add(w[a]);
              m = max(m, (int)w[a]);
              ++k;
              moved = true;
            }
          }
        }
        if (open && q0 >= e && k == cnt && f == fcnt) {
          finish();
          moved = true;
        }
        if (!__any_sync(0xffffffffu, moved)) {
          __nanosleep(20);
          if (give_up()) break;
        }
      }
    }
    if (R == 1) {
      rmax = __reduce_max_sync(0xffffffffu, rmax);
      if (lane == 0 && rmax) atomicMax(&smax[0], rmax);
    }
    __syncthreads();
    for (int x = tid; x < R; x += T)
      if (smax[x]) atomicMax(&V.lev_rounds[(size_t)x * V.lev_stride + (p & 31)], smax[x]);
    // the next level reads words of every block (false once an error was reported)
    if (gridDim.x > 1) ok = grid_sync(V.bar, V.status, V.ns_limit);
    else ok = __syncthreads_and(ok && ld_status(V.status) == 0);
  }
}

// The dataflow kernel's launch for `sites` vertices in R lattices: threads, blocks (one per SM) and
// vertices a block holds; false if the right halves do not fit the blocks' shared memory.
struct FlowShape {
  int threads;
  unsigned grid;
  uint32_t cap, min_tile;
};
// A block owns at least kFlowMinTile vertices: fewer blocks on a small lattice, whose vertices then
// wait for fewer other blocks (L = 256, palette 37: 350 us per colouring with 1024, 358 with 768, 375
// with 512); kFlowThinTile for palettes up to kFlowThin, whose short rows wait for few (exchange
// lattices, palettes of 12 to 17, with 1024, 512 and 256: L = 52 141, 125 and 118 us, L = 128 193, 171
// and 167, L = 256 228, 207 and 205), but a single block up to twice that (L = 24 77 us against
// 84 with two).  A batch, whose palettes are on the device, has 1024.  Blocks of up to kFlowSmall
// vertices run 512 threads (L = 256: 0.45 ms against 0.53 with 1024), larger ones 1024 (1000 x 1337:
// 0.94 ms against 1.01; L = 2304: 4.05 against 4.77).
constexpr uint32_t kFlowMinTile = 1024, kFlowThinTile = 256, kFlowThin = 24, kFlowSmall = 4096;
// g: the palette (0: not known)
inline bool flow_shape(int R, int64_t sites, uint32_t g, FlowShape* sh, cudaError_t* err) {
  static std::atomic<int> smem_of[64];  // per device, once its kernels' limit is raised
  int dev = 0;
  *err = cudaGetDevice(&dev);
  if (*err != cudaSuccess) return false;
  if (dev < 0 || dev >= 64) return false;
  if (smem_of[dev].load() == 0) {
    int b = 0;
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&b, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_kw_flow<512, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               b - 256);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_kw_flow<512, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               b - 256);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_kw_flow<1024, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               b - 256);
    if (e != cudaSuccess) {
      *err = e;
      return false;
    }
    smem_of[dev].store(b - 256);
  }
  const size_t s_smem = (size_t)smem_of[dev].load();
  const int64_t right = (sites + 1) / 2;  // right-half vertices of a level at most
  sh->min_tile = g == 0 || g > kFlowThin    ? kFlowMinTile
                 : right <= 2 * kFlowThinTile ? 2 * kFlowThinTile
                                              : kFlowThinTile;
  sh->grid = (unsigned)std::max<int64_t>(
      1, std::min<int64_t>(num_sms(), (right + sh->min_tile - 1) / sh->min_tile));
  const int64_t own = (right + sh->grid - 1) / sh->grid;
  sh->threads = own <= kFlowSmall ? 512 : 1024;
  const size_t fixed = kw_flow_smem(R, 0, sh->threads);
  if (fixed + 6 * kFlowMinTile > s_smem) return false;
  const int64_t most = std::min<int64_t>(((int64_t)s_smem - (int64_t)fixed) / 6, 65534);
  if (own > most) return false;
  sh->cap = (uint32_t)std::min<int64_t>(most, std::max<int64_t>(own * 5 / 4 + 64, kFlowMinTile + 64));
  return true;
}
inline cudaError_t flow_launch(const FlowView& F, const FlowShape& sh, cudaStream_t st) {
  void* args[] = {(void*)&F};
  // (a single block waits for no other: its lists move by four)
  const void* k = sh.threads == 1024 ? (const void*)k_kw_flow<1024, 2>
                  : sh.grid == 1     ? (const void*)k_kw_flow<512, 4>
                                     : (const void*)k_kw_flow<512, 2>;
  const size_t smem = kw_flow_smem(F.R, sh.cap, sh.threads);
  if (sh.grid == 1) return cudaLaunchKernel(k, dim3(1), dim3(sh.threads), args, smem, st);
  return cudaLaunchCooperativeKernel(k, dim3(sh.grid), dim3(sh.threads), args, smem, st);
}

}  // namespace
}  // namespace sco
