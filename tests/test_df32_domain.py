"""The domain of the float-float and FP32 first decisions (csrc/df32.cuh), on the host: what lies
outside must come out as NaN, so that it is left to the exact decisions."""
import subprocess

import pytest

from paper_1503_03295_gb300 import _build


def run(tmp_path, src):
    nvcc = _build.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    cu, exe = tmp_path / "t.cu", tmp_path / "t"
    cu.write_text(src)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", _build.CSRC, "-o",
                    str(exe), str(cu)], check=True, capture_output=True)
    return subprocess.run([str(exe)], capture_output=True, check=True, text=True).stdout.split()


def test_records_of_spins_out_of_bounds(tmp_path):
    out = run(tmp_path, r"""
#include <cmath>
#include <cstdio>
#include "df32.cuh"
using namespace sco;
int main() {
  const double out[] = {NAN, -NAN, INFINITY, -INFINITY, 1e300, -1e300, 0x1p60, 0x1p64, 2.0, -1.5, 1.001};
  const double in[] = {1.0, -1.0, 1.0 + 0x1p-23, 1.0 + 0x1p-10, 0.0, -0.0, 1e-30, 0.3, -0.9999999999999999};
  int bad = 0;
  for (int k = 0; k < 3; ++k) {
    for (double x : out) {
      const SpinDf d = spin_df(k == 0 ? x : 0.1, k == 1 ? x : 0.2, k == 2 ? x : 0.3, 0);
      bad += !(d.hx != d.hx && d.hy != d.hy && d.hz != d.hz);
    }
    for (double x : in) {
      const SpinDf d = spin_df(k == 0 ? x : 0.1, k == 1 ? x : 0.2, k == 2 ? x : 0.3, 0);
      const double y = k == 0 ? (double)d.hx + d.lx : k == 1 ? (double)d.hy + d.ly : (double)d.hz + d.lz;
      bad += !(std::fabs(y - x) <= 0x1p-47 * std::fabs(x) + 0x1p-60);
    }
  }
  std::printf("%d\n", bad);
}
""")
    assert out == ["0"]
