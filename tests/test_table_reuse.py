"""The temperature-dependent tables (csrc/table.cu) keep their place when the temperature changes: no
second allocation, hence none that could fail and leave a context with freed tables.  The host code is
compiled against counted stand-ins of cudaMalloc and cudaFree and run with no device visible (its kernel
launches then fail, which is not looked at)."""
import os
import subprocess

import pytest

from paper_1503_03295_gb300 import _build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cuda_runtime.h>
static int mallocs = 0, frees = 0, refuse = 0;
template <class T> static cudaError_t test_malloc(T** p, size_t n) {
  ++mallocs;
  *p = refuse ? nullptr : static_cast<T*>(std::malloc(n));
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
static cudaError_t test_free(void* p) { frees += p != nullptr; std::free(p); return cudaSuccess; }
#define cudaMalloc test_malloc
#define cudaFree test_free
#include "table.cu"
#undef cudaMalloc
#undef cudaFree
namespace sco {  // (of scan.cu, for the sorted list only)
size_t scan_tmp_bytes(int64_t) { return 8; }
cudaError_t scan_excl_u32(const uint32_t*, uint32_t*, int64_t, uint64_t*, uint64_t*, cudaStream_t, int64_t*) { return cudaSuccess; }
cudaError_t scan_incl_u64(const uint64_t*, uint64_t*, int64_t, uint64_t*, uint64_t*, cudaStream_t, int64_t*) { return cudaSuccess; }
}
int main() {
  using namespace sco;
  DevParams P{};
  P.Lx = 40; P.Ly = 30; P.N = 1200;
  P.K = 39 + 29 * 79;
  Table t;
  t.K = P.K;
  int64_t launches = 0;
  table_build_xy(P, t, t, nullptr, &launches);
  const Table first = t;
  const int m1 = mallocs, f1 = frees;
  refuse = 1;  // from here on every allocation fails
  P.beta = 3.0;
  table_build_xy(P, t, t, nullptr, &launches);
  const bool same = t.pool == first.pool && t.xy == first.xy && t.pdf == first.pdf && t.far_g == first.far_g && t.far_n == first.far_n;
  const int m2 = mallocs, f2 = frees;
  table_free_xy(t);
  const bool null = !t.pool && !t.xy && !t.qdf && !t.xy32 && !t.sw64 && !t.sw32 && !t.pdf && !t.Ebits && !t.head && !t.near_g && !t.far_g;
  table_build_xy(P, t, t, nullptr, &launches);  // refused
  const bool still = !t.pool && !t.xy && !t.pdf && !t.Ebits;
  std::printf("%d %d %d %d %d %d\n", m1, m2 - m1, f2 - f1, (int)same, (int)null, (int)still);
}
"""


def test_a_change_of_temperature_allocates_nothing(tmp_path):
    nvcc = _build.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([nvcc] + _build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", _build.CSRC, "-I",
                    _build.INCLUDE, "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, check=True, text=True,
                         env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}).stdout
    assert out.split() == ["1", "0", "0", "1", "1", "1"], out
