"""The guides into the decay values (csrc/table.cu, k_guide), on the host: every element writes inside
its guide and every cell gets an entry, also where rounding leaves E a few units out of order (beta D
below 1e-11), and the search's bracket then still holds the first element below a target, to within the
32 units that the search does not trust."""
import subprocess

import pytest

from paper_1503_03295_gb300 import _build

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>
#include <random>
#include "table.cu"
using namespace sco;
static uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
int main() {
  std::mt19937_64 g(5);
  int bad = 0;
  const double rates[] = {0.0, 1e-17, 1e-14, 1e-12, 1e-9, 1e-3, 0.5, 3.0, 200.0, 2000.0};
  for (double bD : rates) for (int K : {1, 2, 100, kNear - 1, kNear, kNear + 1, 9000, 70000}) for (int noise : {0, 3}) {
    std::vector<uint64_t> E(K);
    double w = 0;
    for (int m = 0; m < K; ++m) {
      w += 2 * std::pow((m + 1) / 1.6, -1.5);
      uint64_t b = bD * w < 690 ? bits(std::exp(-bD * w)) : 0;
      if (b && noise) b += (g() % (2 * noise + 1)) - noise;
      E[m] = b < kDecayStart ? b : kDecayStart;
    }
    uint32_t far_n = 64;
    while (far_n < kFarGuide && (int64_t)far_n * 16 < K) far_n *= 2;
    const int64_t nnear = K < kNear ? K : kNear;
    const uint64_t en = E[nnear - 1], el = E[K - 1];
    const int ns = guide_shift(kDecayStart, en, kNearGuide), fs = guide_shift(en, el, far_n);
    std::vector<int64_t> near(kNearGuide + 1, -1), far(far_n + 1, -1);
    for (int64_t m = 0; m <= K; ++m) {
      const bool n = m < nnear;
      const GuideRange r = n ? guide_range(E.data(), m, 0, nnear, kDecayStart, ns, kNearGuide)
                             : guide_range(E.data(), m, nnear, K + 1, en, fs, far_n);
      auto& G = n ? near : far;
      if (r.last >= r.first && (r.first < 0 || r.last >= (int64_t)G.size())) { ++bad; continue; }
      for (int64_t q = r.first; q <= r.last; ++q) G[q] = m;
    }
    for (auto v : near) bad += v < 0;
    for (auto v : far) bad += v < 0;
    // targets around list entries, as the search brackets them
    for (int t = 0; t < 2000; ++t) {
      const uint64_t e = E[g() % K], tb = t % 2 ? e + 40 : (e > 40 ? e - 40 : 0);
      if (tb > kDecayStart) continue;
      int64_t a, b;
      if (tb >= en) {
        const uint64_t q = (kDecayStart - tb) >> ns;
        if (q >= kNearGuide) { ++bad; continue; }
        a = near[q]; b = near[q + 1];
      } else {
        const uint64_t q = (en - tb) >> fs < far_n ? (en - tb) >> fs : far_n - 1;
        a = far[q]; b = far[q + 1];
      }
      while (a < b) { const int64_t mid = (a + b) >> 1; if (E[mid] <= tb) b = mid; else a = mid + 1; }
      int64_t k = 0;
      while (k < K && E[k] > tb) ++k;
      // equal, or left open by the margin
      const bool open = (a < K && E[a] + 32 > tb) || (a > 0 && E[a - 1] < tb + 32);
      bad += a != k && !open;
    }
  }
  std::printf("%d\n", bad);
}
"""


def test_guides_stay_inside(tmp_path):
    nvcc = _build.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC + r"""
namespace sco {
size_t scan_tmp_bytes(int64_t) { return 8; }
cudaError_t scan_excl_u32(const uint32_t*, uint32_t*, int64_t, uint64_t*, uint64_t*, cudaStream_t, int64_t*) { return cudaSuccess; }
cudaError_t scan_incl_u64(const uint64_t*, uint64_t*, int64_t, uint64_t*, uint64_t*, cudaStream_t, int64_t*) { return cudaSuccess; }
}
""")
    subprocess.run([nvcc] + _build.ARCH + ["-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", _build.CSRC,
                    "-I", _build.INCLUDE, "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, check=True, text=True).stdout
    assert out.split() == ["0"], out
