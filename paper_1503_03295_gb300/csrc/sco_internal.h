// sco_internal.h -- host-side declarations shared by the CUDA translation units of the
// SCO library: the launchers each .cu file exports to the C-ABI layer (api.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "df32.cuh"
#include "sco_device.cuh"

namespace sco {

// Device-resident counters of one lattice (one struct per replica).
struct DevCounters {
  unsigned long long n_half;        // surviving half-plane pairs incl. exchange-only bonds
  unsigned long long n_dip;         // surviving dipolar pairs
  unsigned long long ovf_n;         // half-edges beyond the per-site slots
  unsigned long long nnz;           // CSR entries
  unsigned long long guard_fp64;    // decisions re-evaluated in double-double
  unsigned long long guard_fp32;    // decisions re-evaluated in FP64 (FP32-guarded form)
  unsigned int max_degree;          // Delta of the colouring graph
  unsigned int max_degree_dip;      // Delta over dipolar pairs
  unsigned int g;                   // Delta + 1
  unsigned int levels;              // KW levels M
  unsigned int kw_rounds;           // t_R (sum over levels of the deepest dependency chain)
  unsigned int n_colours;           // non-empty classes
  int status;                       // sticky device error (sco_status value), 0 if none
  int ovf_full;                     // the switch wrote more half-edges than the overflow list holds
  double acc[8];                    // observable accumulators
  unsigned int lev_rounds[32];      // deepest dependency chain per KW level
  unsigned int bar[2];              // grid barrier of the persistent kernels
  unsigned int sw_next;             // next unclaimed site of the persistent switch kernel
};

// ---- scan.cu ----
size_t scan_tmp_bytes(int64_t n);
cudaError_t scan_excl_u32(const uint32_t* in, uint32_t* out, int64_t n, uint64_t* tmp,
                          uint64_t* total_dev, cudaStream_t s, int64_t* launches);
cudaError_t scan_incl_u64(const uint64_t* in, uint64_t* out, int64_t n, uint64_t* tmp,
                          uint64_t* total_dev, cudaStream_t s, int64_t* launches);

// ---- table.cu ----
// Guides into the decay bits E for the switch's candidate search (first k with E_k <= tb, on bit
// images).  Near, tb >= e_near = E of the last head element: near[q], q = (bits of 1.0 - tb) >>
// near_shift, is the first k with E_k at or below the largest target of cell q, so the candidate of
// a target in cell q lies in [near[q], near[q + 1]].  Far, below: the same on q = (e_near - tb) >>
// far_shift with far_n cells over the rest of the list.
constexpr int kNear = 2048;       // head of the sorted list kept in shared memory (r <~ 25)
constexpr int kNearGuide = 4096;  // 8 KB; at T = 0.6 D 64 cells per factor of two of E
constexpr uint32_t kFarGuide = 65536;
// Bits of 1.0: the decay value before the first element (W = 0).
constexpr uint64_t kDecayStart = 0x3FF0000000000000ull;
struct SearchHead {
  uint64_t e_near, e_last;
  int32_t near_shift, far_shift;
};
struct Search {
  const uint64_t* E;
  const uint64_t* W;
  const uint32_t* disp;
  const uint16_t* near;
  const uint32_t* far;
  const SearchHead* head;
  int32_t K;
  uint32_t far_n;
};
struct Table {
  int64_t K = 0;
  uint32_t* disp = nullptr;  // packed (dx & 0xFFFF) | (dy << 16), sorted by (r^2, dy, dx)
  uint64_t* W = nullptr;     // inclusive prefix of the integer hazards A_m
  // by list index m: the bits of exp(-beta D 2^-58 W_m), the probability that a walk from
  // the list's start passes m without a candidate (candidate search; temperature-dependent)
  uint64_t* Ebits = nullptr;
  SearchHead* head = nullptr;  // guides into Ebits (see Search)
  uint16_t* near_g = nullptr;
  uint32_t* far_g = nullptr;
  uint32_t far_n = 0;
  double2* xy = nullptr;     // by (|dx|, |dy|): {fl(D c(r^2)), V_max = fl(fl(D A) 2^-59)}
  float2* qdf = nullptr;     // by (|dx|, |dy|): q = -expm1(-2 beta V_max), candidate probability
                             // (float-float)
  float4* xy32 = nullptr;    // by (|dx|, |dy|): FP32 copies {Dc, Vmax, 2 beta Vmax, q}
  Sw64* sw64 = nullptr;      // sweep, by (|dx|, |dy|): FP64 decision constants (see Sw64)
  float4* sw32 = nullptr;    // FP32 sweep: {a1, a3, bvm, 0} of PairDf
  PairDf* pdf = nullptr;     // sweep, by (|dx|, |dy|): the FP64 form's pair constants in float-float
  void* pool = nullptr;      // the one allocation behind the temperature-dependent tables
  size_t pool_bytes = 0;
  int32_t m_nn[2] = {-1, -1};
};
cudaError_t table_build(const DevParams& P, Table& t, cudaStream_t s, int64_t* launches);
// the two halves: the temperature-dependent tables by (|dx|, |dy|) and over the sorted list `list`
// (t's own, or one that several temperatures share), and the sorted list with its hazard prefix
// (depends on Lx, Ly only; synchronises).  The first half's size depends on Lx, Ly only too, so a
// change of temperature fills the tables where they are: it allocates nothing, and nothing is lost
// if it fails (L = 128: 0.172 ms with a pool freed and allocated, 0.045 without).
cudaError_t table_build_xy(const DevParams& P, Table& t, const Table& list, cudaStream_t s,
                           int64_t* launches);
cudaError_t table_build_list(const DevParams& P, Table& t, cudaStream_t s, int64_t* launches);
void table_free(Table& t);
// t's temperature-dependent tables over `list` as the switch searches them
inline Search table_search(const Table& t, const Table& list) {
  return Search{t.Ebits, list.W, list.disp, t.near_g, t.far_g, t.head, (int32_t)list.K, t.far_n};
}
void table_free_xy(Table& t);

// ---- init / observables (spins.cu) ----
// s32, sd: the FP32 and the float-float copies of the spins (either may be null)
cudaError_t spins_init(const DevParams& P, double* s, float4* s32, SpinDf* sd, cudaStream_t st,
                       int64_t* launches);
cudaError_t spins_copies(int64_t N, const double* s, float4* s32, SpinDf* sd, cudaStream_t st,
                         int64_t* launches);
// largest dipolar degree of the current graph into cnt->max_degree_dip
cudaError_t dip_degree_run(const DevParams& P, const uint32_t* row_ptr, const uint32_t* col,
                           DevCounters* cnt, cudaStream_t st, int64_t* launches);
// want_full: the dipolar part of the full energy, by transforms in *work (allocated here when first
// needed or too small, kept by the caller) or, without it, by the direct sum
struct FullWork {
  void* p = nullptr;
  size_t bytes = 0;
};
cudaError_t observables_run(const DevParams& P, const double* s, const uint32_t* row_ptr,
                            const uint32_t* col, const double2* xy, bool have_graph,
                            bool want_full, FullWork* work, DevCounters* cnt, cudaStream_t st,
                            int64_t* launches);
// ---- energy.cu ----
bool full_energy_fft_ok(const DevParams& P);
size_t full_energy_fft_bytes(const DevParams& P);
cudaError_t full_energy_fft(const DevParams& P, const double* s, void* work, double* acc,
                            cudaStream_t st, int64_t* launches);

// ---- switch.cu ----
constexpr int kSlotCap = 32;

// Palettes up to this size can be coloured by the dataflow kernel (kw_flow.cuh): a colour has a byte of
// a word in shared memory.  A batch takes it up to there, a lattice up to flow_max_pal.
constexpr uint32_t kFlowMaxPal = 255;
// With rows of hundreds of entries, read in parts of a list, and chains of hundreds of hops the dataflow
// kernel loses to one kernel per level.  Per colouring, ms, dataflow kernel and kernel per level:
//   L = 64, palette 236: 30.2, 30.1; 202: 19.1, 22.0;  L = 80, 222: 29.7, 29.0;  L = 100, 215: 38.4, 33.7;
//   203: 26.6, 28.0;  L = 128, 223: 50.6, 40.9; 207: 37.4, 37.6;  L = 160, 240: 68.3, 46.8; 210: 41.0, 36.4;
//   195: 35.0, 37.6;  L = 200, 243: 94.1, 63.6; 209: 56.4, 49.1; 199: 33.1, 41.5;  L = 256, 248: 87.4, 74.9;
//   224: 60.7, 63.5;  L = 400, 247: 106, 91; 225: 78.9, 78.7;  L = 512, 243: 126, 109; 234: 98.5, 97.8;  L =
//   700, 246: 135, 126; 233: 114, 122;  L = 1000, 248: 155, 168;  L = 1100 (buckets from 2^20 sites), 248:
//   178, 327.
__host__ __device__ inline uint32_t flow_max_pal(int64_t N) {
  return N < 4608 || N > 800000 ? kFlowMaxPal : N < 50000 ? 208 : 224;
}

// The colouring's level p only looks at neighbours in the same group of g 2^p consecutive sites, for
// the low levels about a sixth of a row, but every row is read at every level.  So the fill
// puts the neighbours in the same group at level near_levels (two lattice rows at most) at the end
// of the row, and the levels up to that one read that end alone.  Sectors read over all levels, by
// the rows that a group spans, against whole rows: 0.56 rows 0.894, 1.1 0.849, 2.25 0.847, 4.5
// 0.870, 9 0.902 (L = 256, T = 0.6 D); 1.4 0.826, 2.9 0.834, 5.8 0.866 (L = 512, T = 0.4 D).
// Per colouring, without and with: L = 2304 3.96 -> 3.77 ms, L = 1024 T = 0.4 D 1.21 -> 1.15; groups of
// up to one row 3.81 and 1.16, four rows 3.78 and 1.15.
// max_pal: the largest palette that the dataflow kernel will take.
__host__ __device__ inline unsigned near_levels(uint32_t g, uint32_t Lx, uint32_t max_pal) {
  unsigned p = 0;
  if (g <= max_pal)
    while ((g << (p + 1)) <= 2 * Lx) ++p;
  return p;
}
// Where the fill puts the neighbours of a lattice: cur counts a row's far (low 16 bits) and near
// entries, which stay below 2^16 for palettes of the dataflow kernel; larger ones have no near part
// and count in 32 bits.
// On larger lattices (kSplitSites), rows of palettes beyond the dataflow kernel hold the smaller
// neighbours first, then the larger ones in the order of their slots, by distance: the lanes of a warp,
// at neighbouring sites, then look at the words of neighbouring sites at a time.  The cursors count the
// smaller neighbours only.  Per colouring in this order and all by atomic order: L = 300, palette 300 517
// and 552 ms, L = 256 804 and 890, L = 200 461 and 472, L = 128 274 and 271, L = 64 (palette 421) 1717 and
// 1331 (there the spread makes neighbouring lanes wait for different vertices).
constexpr int64_t kSplitSites = 1 << 15;
struct RowFill {
  uint32_t group, mask;  // sites per group (0: no near part), far count in a cursor
  bool split;            // smaller neighbours, then larger ones
};
__host__ __device__ inline RowFill row_fill(uint32_t g, uint32_t Lx, int64_t N, uint32_t max_pal) {
  const unsigned p = near_levels(g, Lx, max_pal);
  return p ? RowFill{g << p, 0xFFFFu, false}
           : RowFill{0, 0xFFFFFFFFu, g > max_pal && N >= kSplitSites};
}
struct SwitchBufs {
  uint32_t* hslot;  // N * kSlotCap upper neighbours (j | flag) per site
  uint32_t* hcnt;   // N half-degree per site (the fill counts the overflow half-edges down)
  uint32_t* indeg;  // N lower-neighbour count per site
  uint32_t* deg;    // N + 1
  uint32_t* lcur;   // N row cursors, then what the rows hold (see RowFill)
  uint32_t* ovf;    // 2 * ovf_cap (i, j | flag)
  uint32_t ovf_cap;
  uint64_t* scan_tmp;
};
cudaError_t switch_run(const DevParams& P, const Table& t, const double* s, const float4* s32,
                       const SpinDf* sd, int precision, uint32_t epoch, SwitchBufs& b, DevCounters* cnt,
                       cudaStream_t st, int64_t* launches);
cudaError_t csr_scan(const DevParams& P, SwitchBufs& b, uint32_t* row_ptr, DevCounters* cnt,
                     cudaStream_t st, int64_t* launches);
// A row holds its far neighbours from its start and its near ones from its end, each in the order of
// their atomic slots (no result depends on the order inside a row).
cudaError_t csr_fill(const DevParams& P, const SwitchBufs& b, uint32_t g, const uint32_t* row_ptr,
                     uint32_t* col, bool has_overflow, DevCounters* cnt, cudaStream_t st,
                     int64_t* launches);
// w.p[0 .. nnz) = col[first ..] with every row sorted by neighbour index (the documented layout of the
// getters), row_ptr[0] = first; also records the largest dipolar degree in cnt.  The caller keeps the
// workspace up to kSortKeep entries (an allocation took up to 0.17 of a batch getter's 0.23 ms) and
// releases a larger one after the copy to the host.
constexpr uint64_t kSortKeep = 1ull << 24;
struct SortWork {
  uint32_t* p = nullptr;
  uint64_t cap = 0;
  void release() {
    cudaFree(p);
    p = nullptr;
    cap = 0;
  }
};
cudaError_t csr_sorted_copy(const DevParams& P, const uint32_t* row_ptr, const uint32_t* col,
                            uint32_t first, uint64_t nnz, SortWork& w, DevCounters* cnt, cudaStream_t st,
                            int64_t* launches);

// ---- colour.cu ----
struct ColourBufs {
  unsigned long long* word;  // N packed (level tag, round, colour)
  uint8_t* col8;     // N colour (low byte), kept beside the words for the neighbour gathers
  uint32_t* blk;     // N neighbour each unfinished vertex waits for (0xFFFFFFFF: none)
  uint32_t* colour;  // N final colours
  uint32_t* hist;    // g + 1
  uint32_t* off;     // g + 1
  uint32_t* cursor;  // g
  uint32_t* perm;    // N
  uint32_t* tile_cnt;  // (colour, tile, degree bin) counts (+1), scanned in place
  uint64_t* scan_tmp;
  uint32_t* bcnt;    // 32 x palette KW bucket sizes per level
  uint32_t* meta;    // 6 words: one-lattice view of the persistent colouring kernel
  unsigned long long* imask;  // N per-level vertex records of the colouring kernel
  uint32_t* imeta;            // N
  uint32_t* ilist;            // 32 N (kItemList per record)
  uint32_t* boff;             // kKwSplitBlocks x 64: per (block, colour) bucket offsets of the
                              // split record build (null: records built inside k_kw_bcr)
};
constexpr int kKwSplitBlocks = 2048;
constexpr uint32_t kMaxStablePalette = 12288;  // palettes up to this size get stable classes
constexpr int64_t kClassTileSites = 2048;
// rows: the cursors that csr_fill left; ns_limit: bound of every device-side wait of the colouring
// kernels (SCO_ETIMEOUT after it)
cudaError_t kw_run(const DevParams& P, const uint32_t* row_ptr, const uint32_t* col, const uint32_t* rows,
                   uint32_t g, int variant, ColourBufs& b, DevCounters* cnt,
                   unsigned long long ns_limit, cudaStream_t st, int64_t* launches);
cudaError_t bucket_run(const DevParams& P, uint32_t g, const uint32_t* row_ptr, ColourBufs& b,
                       DevCounters* cnt, cudaStream_t st, int64_t* launches);

// ---- sweep.cu ----
// s32 and prop32 (FP32-guarded form) or sd and propd (FP64 form): the working copies of the spins and
// the proposals of the step; the others are null.
struct SweepBufs {
  double* s;
  float4* s32;
  SpinDf* sd;
  const uint32_t* row_ptr;
  const uint32_t* col;
  const uint32_t* perm;
  const uint32_t* off;
  double4_32a* prop;
  SpinDf* propd;
  float4* prop32;
  uint8_t* acc;
};
cudaError_t sweep_run(const DevParams& P, const Table& t, const SweepBufs& b, uint32_t g,
                      uint64_t step, int precision, DevCounters* cnt, unsigned long long ns_limit,
                      cudaStream_t st, int64_t* launches);

// ---- stats.cu ----
// Graph diagnostics (see sco_get_graph_stats); copies 2 nb + 1 counts (survived, pairs, cross)
// to h_counts and 6 + g + nb doubles (summary, Delta R per colour, P_survive) to h_out, then
// synchronises.
cudaError_t graph_stats_run(const DevParams& P, const uint32_t* disp, const uint32_t* row_ptr,
                            const uint32_t* col, const uint32_t* colour, uint32_t g, int cx,
                            int cy, int nb, cudaStream_t st, int64_t* launches,
                            unsigned long long* h_counts, double* h_out);

int num_sms();

}  // namespace sco
