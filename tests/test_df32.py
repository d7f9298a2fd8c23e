"""Float-float arithmetic of the FP64 form's decisions (csrc/df32.cuh), compiled for the host and
held against long double: the bounds that the decisions carry in their margins."""
import os
import subprocess

import pytest

from paper_1503_03295_gb300 import _build

SRC = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "df32.cuh"
using namespace sco;
typedef long double L;
int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(0, 1);
  std::normal_distribution<double> G(0, 1);
  L em = 0, ep = 0, ey = 0, fm = 0, fy = 0;
  for (long i = 0; i < 3000000; ++i) {
    const double y0 = i % 4 == 0 ? U(g) * 0.42 : i % 4 == 1 ? U(g) * 20
                    : i % 4 == 2 ? std::exp(-U(g) * 60) : std::exp(U(g) * 9);
    const float h = (float)y0, l = (float)(y0 - h);
    if (!(h < 8192.f)) continue;
    const L Y = (L)h + l;
    int k;
    const df m = df_expm1_scaled({h, l}, k), p = df_one_minus_exp_neg({h, l});
    // given y: y itself to 2^-42 of its size (ln 2 in three parts)
    const L x = k == 0 ? expm1l(Y) : expl(Y - k * logl(2.0L)) - ldexpl(1, -k);
    em = fmaxl(em, fabsl((L)m.h + m.l - x) - Y * 0x1p-42L > 0 ? fabsl(((L)m.h + m.l - x) / x) : 0);
    {
      int kf;
      const float m32 = f32_expm1_scaled(h, kf);
      const L H = h, x32 = kf == 0 ? expm1l(H) : expl(H - kf * logl(2.0L)) - ldexpl(1, -kf);
      if (h < 60.f) fm = fmaxl(fm, fabsl((m32 - x32) / x32));
    }
    ep = fmaxl(ep, fabsl(((L)p.h + p.l + expm1l(-Y)) / expm1l(-Y)));
  }
  for (long i = 0; i < 1000000; ++i) {
    int dx = (int)std::exp(U(g) * 7.7) - 1, dy = (int)std::exp(U(g) * 7.7) - 1;
    if (i % 3 == 0) dx %= 4, dy %= 4;
    if (dx == 0 && dy == 0) dx = 1;
    const double r2 = (double)dx * dx + (double)dy * dy, c = 1 / (r2 * r2 * std::sqrt(r2));
    const double beta = std::exp(U(g) * 6 - 2), a1 = beta * (c * r2), a3 = beta * (3 * c);
    const double A = (double)(unsigned long long)(0x1p60 / (r2 * std::sqrt(r2)) * (1 + 0x1p-50)) + 1;
    const double bvm = beta * (A * 0x1p-59);
    double S[2][3];
    for (int k = 0; k < 2; ++k) {
      for (int j = 0; j < 3; ++j) S[k][j] = G(g);
      if (i % 2) {  // near the bond: V near Vmax
        const double rr = std::sqrt(r2), e = std::exp(-U(g) * 12), o = k ? -1 : 1;
        S[k][0] = o * dx / rr + e * S[k][0];
        S[k][1] = o * dy / rr + e * S[k][1];
        S[k][2] *= e;
      }
      const double n = std::sqrt(S[k][0] * S[k][0] + S[k][1] * S[k][1] + S[k][2] * S[k][2]);
      for (int j = 0; j < 3; ++j) S[k][j] /= n;
    }
    const df d1 = df_split_const(a1), d3 = df_split_const(a3), dv = df_split_const(bvm);
    const PairDf t = {d1.h, d1.l, d3.h, d3.l, dv.h, dv.l, (float)dx, (float)dy};
    const SpinDf a = spin_df(S[0][0], S[0][1], S[0][2], 0), b = spin_df(S[1][0], S[1][1], S[1][2], 0);
    const df y = df_pair_y(t, df_field(t, t.ax, t.ay, b), a);
    const L ss = (L)S[0][0] * S[1][0] + (L)S[0][1] * S[1][1] + (L)S[0][2] * S[1][2];
    const L pa = (L)S[0][0] * dx + (L)S[0][1] * dy, pb = (L)S[1][0] * dx + (L)S[1][1] * dy;
    const L V = (L)c * ((L)r2 * ss - 3 * pa * pb);
    float gx, gy, gz;
    f32_field((float)a1, (float)a3, t.ax, t.ay, (float)S[1][0], (float)S[1][1], (float)S[1][2], gx, gy,
              gz);
    const float y32 = f32_y((float)bvm, gx, gy, gz, (float)S[0][0], (float)S[0][1], (float)S[0][2]);
    fy = fmaxl(fy, fabsl((L)y32 - (L)beta * ((L)A * 0x1p-59L - V)) / (L)a1);
    ey = fmaxl(ey, fabsl((L)y.h + y.l - (L)beta * ((L)A * 0x1p-59L - V)) / (L)a1);
  }
  std::printf("%.3f %.3f %.3f %.3f %.3f\n", (double)log2l(em), (double)log2l(ep), (double)log2l(ey),
              (double)log2l(fm), (double)log2l(fy));
}
"""


def test_bounds(tmp_path):
    nvcc = _build.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", _build.CSRC,
                    "-o", str(exe), str(src)], check=True, capture_output=True)
    em, ep, ey, fm, fy = map(float, subprocess.run([str(exe)], capture_output=True, check=True,
                                                   text=True).stdout.split())
    # 2^-31: kDfExpRelErr (relative, e^y - 1 and 1 - e^-y); 2^-40: kYRelErr (of a1)
    assert em <= -31.0 and ep <= -31.0 and ey <= -40.0, (em, ep, ey)
    # the plain FP32 terms: 2^-20 kE32RelErr, 2^-18 kY32RelErr
    assert fm <= -20.0 and fy <= -18.0, (fm, fy)
    print(em, ep, ey, fm, fy)
