// energy.cu -- the full dipolar energy of Eq. (6) as a correlation, by FP64 Fourier transforms.
//
// E = 1/2 sum_d sum_i S_i . M(d) S_(i+d) with M(d) = D c(r^2) (r^2 1 - 3 d d^T), d = (dx, dy, 0).
// On the lattice padded to a power of two >= 2 L in each direction no displacement wraps, and with
// S(k) and M(k) the transforms E = 1/(2 P) sum_k S(k)* . M(k) S(k), P the padded points.  M is even
// in d, so its four components have real transforms and go in pairs through two complex transforms
// (xx + i yy, zz + i xy); the spins take two (x + i y, z).
//
// The direct sum's N^2 / 2 pairs (each with an FP64 square root and division) took 212 ms at N =
// 65,536 on the FP64 pipe, and 0.38 ms at N = 256; the four transforms of 512 x 512 points are 0.1
// GFLOP: 0.22 ms at N = 65,536, 0.02 ms at N = 256 (times beside the other observables').  Two launches, bound
// by shared-memory latency: transforms along the longer side (a block per line), then along the
// shorter one, a block per pair of columns +-k of all four arrays, which also sums the energy (the
// transformed arrays never go back to memory).
#include <cmath>
#include <cstdint>

#include "sco_internal.h"

namespace sco {

namespace {

constexpr int kFftThreads = 256;
// lattice side: lines of at most 2048 points, two of them in a block's shared memory
constexpr int kFftMaxSide = 1024;

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// In-place decimation-in-frequency transforms of `lines` lines of n = 2^logn points in shared memory
// (line l at a + l n): position q ends with frequency bit_reverse(q).  tw[j] = exp(-2 pi i j / n).
__device__ void fft_lines(double2* a, int logn, int lines, const double2* tw) {
  const int n = 1 << logn;
  for (int h = n >> 1, s = 1; h > 0; h >>= 1, s <<= 1) {
    for (int q = threadIdx.x; q < lines * (n >> 1); q += blockDim.x) {
      const int l = q >> (logn - 1), b = q & ((n >> 1) - 1);
      const int j = b & (h - 1), i = ((b - j) << 1) + j;
      double2* x = a + (size_t)l * n + i;
      const double2 u = x[0], v = x[h];
      x[0] = make_double2(u.x + v.x, u.y + v.y);
      x[h] = cmul(make_double2(u.x - v.x, u.y - v.y), tw[j * s]);
    }
    __syncthreads();
  }
}
__device__ void fft_twiddles(double2* tw, int logn) {
  const int n = 1 << logn;
  for (int j = threadIdx.x; j < n / 2; j += blockDim.x) {
    double s, c;
    sincospi(-2.0 * j / n, &s, &c);
    tw[j] = make_double2(c, s);
  }
}

// The lattice with its longer side A (points a, site stride sa) and its shorter one B.
struct FftShape {
  int na, nb;    // sides
  int la, lb;    // log2 of the padded sides
  int64_t sa, sb;
  int swap;      // A is the y side
};

// Transforms along A.  Block b < nb: the spins of line b, two arrays; then the couplings at signed
// displacement db for every padded line, two arrays.  out: four arrays of Pb x Pa points (spin lines
// b < nb only).
__global__ void __launch_bounds__(kFftThreads) k_fft_a(const DevParams P, const FftShape F,
                                                       const double* __restrict__ s,
                                                       double2* __restrict__ out) {
  extern __shared__ double2 fs[];
  const int n = 1 << F.la, pb = 1 << F.lb;
  double2* tw = fs + 2 * n;
  const int line = blockIdx.x;
  const bool spins = line < F.nb;
  const int row = spins ? line : line - F.nb;
  const int db = row <= pb / 2 ? row : row - pb;
  if (!spins && (db >= F.nb || -db >= F.nb)) {  // no pair at this displacement
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
      out[((size_t)2 * pb + row) * n + q] = make_double2(0.0, 0.0);
      out[((size_t)3 * pb + row) * n + q] = make_double2(0.0, 0.0);
    }
    return;
  }
  fft_twiddles(tw, F.la);
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    double2 u = make_double2(0.0, 0.0), v = u;
    if (spins) {
      if (q < F.na) {
        const int64_t i = q * F.sa + row * F.sb;
        u = make_double2(s[i], s[P.N + i]);
        v = make_double2(s[2 * P.N + i], 0.0);
      }
    } else {
      const int da = q <= n / 2 ? q : q - n;
      if (da < F.na && -da < F.na && (da != 0 || db != 0)) {
        const double dx = F.swap ? db : da, dy = F.swap ? da : db;
        const int64_t r2 = (int64_t)da * da + (int64_t)db * db;
        const double c = P.D * coupling_c(r2), q2 = (double)r2;
        u = make_double2(c * (q2 - 3.0 * dx * dx), c * (q2 - 3.0 * dy * dy));
        v = make_double2(c * q2, -3.0 * c * dx * dy);
      }
    }
    fs[q] = u;
    fs[n + q] = v;
  }
  __syncthreads();
  fft_lines(fs, F.la, 2, tw);
  const size_t o = spins ? 0 : 2;
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    out[((o + 0) * pb + row) * n + q] = fs[q];
    out[((o + 1) * pb + row) * n + q] = fs[n + q];
  }
}

// Transforms along B of the columns at frequencies +-k of A (block k = 0 .. Pa/2; the two coincide
// for k = 0 and Pa/2), and the energy of their points: with f = FT(Sx + i Sy) at K and g = f at -K,
// X = (f + g*) / 2, Y = (f - g*) / (2 i).
__global__ void __launch_bounds__(kFftThreads) k_fft_b(const FftShape F,
                                                       const double2* __restrict__ in,
                                                       double* __restrict__ acc) {
  extern __shared__ double2 fs[];
  const int na = 1 << F.la, n = 1 << F.lb;
  double2* tw = fs + 8 * n;
  const unsigned k = blockIdx.x;
  const unsigned ca = __brev(k) >> (32 - F.la), cb = __brev((na - k) & (na - 1)) >> (32 - F.la);
  fft_twiddles(tw, F.lb);
  for (int q = threadIdx.x; q < 8 * n; q += blockDim.x) {
    const int a = q & 7, y = q >> 3;  // array and column side: neighbouring threads, one row
    const int arr = a >> 1;
    double2 v = make_double2(0.0, 0.0);
    if (arr >= 2 || y < F.nb) v = in[((size_t)arr * n + y) * na + (a & 1 ? cb : ca)];
    fs[(size_t)a * n + y] = v;
  }
  __syncthreads();
  fft_lines(fs, F.lb, 8, tw);
  double e = 0.0;
  const double w = ca == cb ? 0.5 : 1.0;  // a column that is its own partner comes up twice
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const unsigned m = __brev((unsigned)q) >> (32 - F.lb);
    const int r = (int)(__brev((n - m) & (n - 1)) >> (32 - F.lb));  // position of frequency -m
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const double2 f = fs[(size_t)side * n + q], g = fs[(size_t)(1 - side) * n + r];
      const double2 z = fs[(size_t)(2 + side) * n + q];
      const double2 m1 = fs[(size_t)(4 + side) * n + q], m2 = fs[(size_t)(6 + side) * n + q];
      const double2 X = make_double2(0.5 * (f.x + g.x), 0.5 * (f.y - g.y));
      const double2 Y = make_double2(0.5 * (f.y + g.y), 0.5 * (g.x - f.x));
      e += w * (m1.x * (X.x * X.x + X.y * X.y) + m1.y * (Y.x * Y.x + Y.y * Y.y) +
                m2.x * (z.x * z.x + z.y * z.y) + 2.0 * m2.y * (X.x * Y.x + X.y * Y.y));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(acc, e * (0.5 / ((double)na * n)));
}

}  // namespace

// log2 of the padded side; 0 for a side of one site needs one point
static int padded_log2(int side) {
  int l = 1;
  while ((1 << l) < 2 * side) ++l;
  return l;
}

static FftShape fft_shape(const DevParams& P) {
  FftShape F{};
  F.swap = P.Ly > P.Lx ? 1 : 0;
  F.na = F.swap ? P.Ly : P.Lx;
  F.nb = F.swap ? P.Lx : P.Ly;
  F.sa = F.swap ? P.Lx : 1;
  F.sb = F.swap ? 1 : P.Lx;
  F.la = padded_log2(F.na);
  F.lb = padded_log2(F.nb);
  return F;
}

bool full_energy_fft_ok(const DevParams& P) {
  return P.N <= 65536 && P.Lx <= kFftMaxSide && P.Ly <= kFftMaxSide;
}
size_t full_energy_fft_bytes(const DevParams& P) {
  const FftShape F = fft_shape(P);
  return ((size_t)4 << (F.la + F.lb)) * sizeof(double2);
}

cudaError_t full_energy_fft(const DevParams& P, const double* s, void* work, double* acc,
                            cudaStream_t st, int64_t* launches) {
  const FftShape F = fft_shape(P);
  const int pa = 1 << F.la, pb = 1 << F.lb;
  const size_t sha = ((size_t)2 * pa + pa / 2) * sizeof(double2);
  const size_t shb = ((size_t)8 * pb + pb / 2) * sizeof(double2);
  cudaError_t e = cudaSuccess;
  if (sha > 48 * 1024)
    e = cudaFuncSetAttribute(k_fft_a, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sha);
  if (e == cudaSuccess && shb > 48 * 1024)
    e = cudaFuncSetAttribute(k_fft_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shb);
  if (e != cudaSuccess) return e;
  double2* buf = static_cast<double2*>(work);
  k_fft_a<<<(unsigned)(F.nb + pb), kFftThreads, sha, st>>>(P, F, s, buf);
  k_fft_b<<<(unsigned)(pa / 2 + 1), kFftThreads, shb, st>>>(F, buf, acc);
  *launches += 2;
  return cudaGetLastError();
}

}  // namespace sco
