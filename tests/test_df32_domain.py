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


def test_weak_pairs(tmp_path):
    # y = beta (Vmax - V) of pairs so weak that FP32 runs out of exponents: within kYRelErr a1 (FP32: kY32RelErr
    # a1) wherever it is above kYMin
    out = run(tmp_path, r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "df32.cuh"
using namespace sco;
typedef long double L;
int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(0, 1);
  std::normal_distribution<double> G(0, 1);
  L ey = 0, fy = 0;
  long n = 0;
  for (long i = 0; i < 2000000; ++i) {
    const int dx = (int)std::exp(U(g) * 10.39), dy = (int)std::exp(U(g) * 10.39);
    const double r2 = (double)dx * dx + (double)dy * dy, c = 1 / (r2 * r2 * std::sqrt(r2));
    const double beta = std::exp2(-U(g) * 90), a1 = beta * (c * r2), a3 = beta * (3 * c);
    const double A = (double)(unsigned long long)(0x1p60 / (r2 * std::sqrt(r2)) * (1 + 0x1p-50)) + 1;
    const double bvm = beta * (A * 0x1p-59);
    double S[2][3];
    for (auto& s : S) {
      for (double& x : s) x = G(g);
      const double m = std::sqrt(s[0] * s[0] + s[1] * s[1] + s[2] * s[2]);
      for (double& x : s) x /= m;
    }
    const df d1 = df_split_const(a1), d3 = df_split_const(a3), dv = df_split_const(bvm);
    const PairDf t = {d1.h, d1.l, d3.h, d3.l, dv.h, dv.l, (float)dx, (float)dy};
    const SpinDf a = spin_df(S[0][0], S[0][1], S[0][2], 0), b = spin_df(S[1][0], S[1][1], S[1][2], 0);
    const df y = df_pair_y(t, df_field(t, t.ax, t.ay, b), a);
    const L ss = (L)S[0][0] * S[1][0] + (L)S[0][1] * S[1][1] + (L)S[0][2] * S[1][2];
    const L pa = (L)S[0][0] * dx + (L)S[0][1] * dy, pb = (L)S[1][0] * dx + (L)S[1][1] * dy;
    const L Y = (L)beta * ((L)A * 0x1p-59L - (L)c * ((L)r2 * ss - 3 * pa * pb));
    float gx, gy, gz;
    f32_field((float)a1, (float)a3, t.ax, t.ay, (float)S[1][0], (float)S[1][1], (float)S[1][2], gx, gy, gz);
    const float y32 = f32_y((float)bvm, gx, gy, gz, (float)S[0][0], (float)S[0][1], (float)S[0][2]);
    if (y.h > kYMin) ey = fmaxl(ey, fabsl((L)y.h + y.l - Y) / (L)a1), ++n;
    if (y32 > kYMin) fy = fmaxl(fy, fabsl((L)y32 - Y) / (L)a1);
  }
  std::printf("%d %d %d\n", ey <= kYRelErr, fy <= kY32RelErr, n > 100000);
}
""")
    assert out == ["1", "1", "1"], out


def test_folds(tmp_path):
    # an exponent of up to 2^20 as k ln 2 + y' with y' in the exponential's range
    out = run(tmp_path, r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "df32.cuh"
using namespace sco;
typedef long double L;
int main() {
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> U(0, 1);
  L e = 0, f = 0;
  int bad = 0;
  for (long i = 0; i < 2000000; ++i) {
    const double y0 = (i & 1 ? -1 : 1) * std::exp2(13 + 7 * U(g)) * 0.999999;
    const float h = (float)y0, l = (float)(y0 - h);
    int k, kf;
    const df y = df_fold({h, l}, k);
    const float y32 = f32_fold(h, kf);
    if (h > 0) {  // as the pair terms use it
      int kk, ke;
      const df r = df_fold({h, l}, kk, 128.f);
      e = fmaxl(e, fabsl((L)r.h + r.l + kk * logl(2.0L) - ((L)h + l)) / fabsl((L)h));
      const df m = df_expm1_scaled(r, ke);
      const L x = expl((L)h + l - (kk + ke) * logl(2.0L));  // (e^y - 1) 2^-k
      bad += !(fabsl((L)m.h + m.l - x) <= (0x1p-31L + 0x1p-42L * h) * x) || ke < 127;
    }
    e = fmaxl(e, fabsl((L)y.h + y.l + k * logl(2.0L) - ((L)h + l)) / fabsl((L)h));
    f = fmaxl(f, fabsl((L)y32 + kf * logl(2.0L) - (L)h) / fabsl((L)h));
    const float s = i & 1 ? -1.f : 1.f;
    bad += !(s * y.h > -0.1f && s * y.h < 5679.f && s * y32 > -0.1f && s * y32 < 5679.f) || k % 8192 != 0 || kf != k;
  }
  std::printf("%d %d %d\n", e <= 0x1p-43L, f <= 0x1p-23L, bad);
}
""")
    assert out == ["1", "1", "0"], out
