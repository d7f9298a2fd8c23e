"""The error bounds of the first decisions (csrc/df32.cuh) over the whole range that they admit, on the host:
the exponentials up to y = 8192 without exclusions, pair terms up to beta = e^9, and a running error analysis of
the pair term (each rounding's own bound added up along the computation), which must stay below twice the
stated bound, since the decisions double it."""
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
static const double u = 0x1p-24;
// a value h + l with a bound on its distance from the exact one
struct R { double h, l, e; };
static R rd(df d, double e) { return {d.h, d.l, e}; }
static double mag(const R& a) { return std::fabs(a.h) + std::fabs(a.l) + a.e; }
static R two(R a, R b, double sg) {  // df_add, df_sub
  const df s = df_two_sum((float)a.h, (float)(sg * b.h));
  const float t = (float)a.l + (float)(sg * b.l), l = s.l + t;
  return {s.h, l, a.e + b.e + u * std::fabs(t) + u * std::fabs(l)};
}
static R mulr(R a, R b) {  // df_mul
  const float p = (float)a.h * (float)b.h, e = df_fma((float)a.h, (float)b.h, -p);
  const float m = df_fma((float)a.h, (float)b.l, e), l = df_fma((float)a.l, (float)b.h, m);
  return {p, l, u * std::fabs(m) + u * std::fabs(l) + std::fabs(a.l * b.l) + mag(a) * b.e + mag(b) * a.e};
}
static R mulf(R a, float f) {  // df_mul_f
  const float p = (float)a.h * f, e = df_fma((float)a.h, f, -p), l = df_fma((float)a.l, f, e);
  return {p, l, u * std::fabs(l) + std::fabs(f) * a.e};
}
int main() {
  std::mt19937_64 g(29);
  std::uniform_real_distribution<double> U(0, 1);
  std::normal_distribution<double> G(0, 1);
  L em = 0, ep = 0, fm = 0, ey = 0, fy = 0;
  double er = 0, fr = 0;
  for (long i = 0; i < 4000000; ++i) {
    const double y0 = i % 4 == 0 ? U(g) * 0.42 : i % 4 == 1 ? U(g) * 60 : i % 4 == 2 ? std::exp(-U(g) * 41) : U(g) * 8191.9;
    const float h = (float)y0, l = (float)(y0 - h);
    const L Y = (L)h + l;
    int k, kf;
    const df m = df_expm1_scaled({h, l}, k), p = df_one_minus_exp_neg({h, l});
    const L x = k == 0 ? expm1l(Y) : expl(Y - k * logl(2.0L)) - ldexpl(1, -k);
    em = fmaxl(em, fabsl(((L)m.h + m.l - x) / x));
    ep = fmaxl(ep, fabsl(((L)p.h + p.l + expm1l(-Y)) / expm1l(-Y)));
    const float m32 = f32_expm1_scaled(h, kf);
    const L x32 = kf == 0 ? expm1l((L)h) : expl(h - kf * logl(2.0L)) - ldexpl(1, -kf);
    fm = fmaxl(fm, fabsl((m32 - x32) / x32));
  }
  for (long i = 0; i < 3000000; ++i) {
    int dx = (int)std::exp(U(g) * 9) - 1, dy = (int)std::exp(U(g) * 9) - 1;
    if (i % 3 == 0) dx %= 6, dy %= 6;
    if (dx == 0 && dy == 0) dx = 1;
    const double r2 = (double)dx * dx + (double)dy * dy, c = 1 / (r2 * r2 * std::sqrt(r2));
    const double beta = std::exp(U(g) * 13 - 4), a1 = beta * (c * r2), a3 = beta * (3 * c);
    const double A = (double)(unsigned long long)(0x1p60 / (r2 * std::sqrt(r2)) * (1 + 0x1p-50)) + 1;
    const double bvm = beta * (A * 0x1p-59);
    double S[2][3];
    for (int k = 0; k < 2; ++k) {
      for (int j = 0; j < 3; ++j) S[k][j] = G(g);
      if (i % 4) {  // along the bond or across it, more or less
        const double rr = std::sqrt(r2), e = std::exp(-U(g) * 12), o = U(g) < 0.5 ? -1 : 1;
        const double bx = i % 4 == 3 ? -dy : dx, by = i % 4 == 3 ? dx : dy;
        S[k][0] = o * bx / rr + e * S[k][0];
        S[k][1] = o * by / rr + e * S[k][1];
        S[k][2] *= e;
      }
      const double n = std::sqrt(S[k][0] * S[k][0] + S[k][1] * S[k][1] + S[k][2] * S[k][2]);
      for (int j = 0; j < 3; ++j) S[k][j] /= n;
    }
    const df d1 = df_split_const(a1), d3 = df_split_const(a3), dv = df_split_const(bvm);
    const PairDf t = {d1.h, d1.l, d3.h, d3.l, dv.h, dv.l, (float)dx, (float)dy};
    const SpinDf s = spin_df(S[0][0], S[0][1], S[0][2], 0), b = spin_df(S[1][0], S[1][1], S[1][2], 0);
    const df y = df_pair_y(t, df_field(t, t.ax, t.ay, b), s);
    const L ss = (L)S[0][0] * S[1][0] + (L)S[0][1] * S[1][1] + (L)S[0][2] * S[1][2];
    const L pa = (L)S[0][0] * dx + (L)S[0][1] * dy, pb = (L)S[1][0] * dx + (L)S[1][1] * dy;
    const L X = (L)beta * ((L)A * 0x1p-59L - (L)c * ((L)r2 * ss - 3 * pa * pb));
    ey = fmaxl(ey, fabsl((L)y.h + y.l - X) / (L)a1);
    float gx, gy, gz;
    f32_field((float)a1, (float)a3, t.ax, t.ay, (float)S[1][0], (float)S[1][1], (float)S[1][2], gx, gy, gz);
    const float y32 = f32_y((float)bvm, gx, gy, gz, (float)S[0][0], (float)S[0][1], (float)S[0][2]);
    fy = fmaxl(fy, fabsl((L)y32 - X) / (L)a1);
    // running errors: constants rounded in FP64 (4 units) and split, spins split
    const double kc = 0x1p-48 + 4 * 0x1p-53, ks = 0x1p-47;
    const R A1 = rd(d1, kc * a1), A3 = rd(d3, kc * a3), BV = rd(dv, kc * bvm);
    auto comp = [&](float hh, float ll, double x) { return R{hh, ll, ks * std::fabs(x) + 0x1p-60}; };
    const R sx = comp(s.hx, s.lx, S[0][0]), sy = comp(s.hy, s.ly, S[0][1]), sz = comp(s.hz, s.lz, S[0][2]);
    const R bx = comp(b.hx, b.lx, S[1][0]), by = comp(b.hy, b.ly, S[1][1]), bz = comp(b.hz, b.lz, S[1][2]);
    const R q = two(mulf(bx, t.ax), mulf(by, t.ay), 1), w = mulr(A3, q);
    const R fx = two(mulr(A1, bx), mulf(w, t.ax), -1), fy_ = two(mulr(A1, by), mulf(w, t.ay), -1), fz = mulr(A1, bz);
    R Y = two(two(two(BV, mulr(fx, sx), -1), mulr(fy_, sy), -1), mulr(fz, sz), -1);
    const double low = std::fabs(Y.h) + std::fabs(Y.l);
    er = std::fmax(er, (Y.e + u * u * low) / a1);  // (and the last renormalisation)
    // plain FP32: spins and constants rounded, every operation u of its result
    {
      const double k1 = u, B0 = std::fabs(S[1][0]), B1 = std::fabs(S[1][1]), B2 = std::fabs(S[1][2]);
      const double p1 = B1 * dy, pe = k1 * p1 + u * p1, q0 = std::fabs(S[1][0] * dx + S[1][1] * dy), qe = pe + k1 * B0 * dx + u * (q0 + pe);
      const double w0 = a3 * q0, we = a3 * qe + k1 * w0 + u * w0;
      const double gx0 = std::fabs(a1 * S[1][0] - a3 * (S[1][0] * dx + S[1][1] * dy) * dx), gxe = we * dx + u * w0 * dx + 2 * k1 * a1 * B0 + u * gx0;
      const double gy0 = std::fabs(a1 * S[1][1] - a3 * (S[1][0] * dx + S[1][1] * dy) * dy), gye = we * dy + u * w0 * dy + 2 * k1 * a1 * B1 + u * gy0;
      const double gz0 = a1 * B2, gze = 3 * k1 * gz0;
      const double s0 = std::fabs(S[0][0]), s1 = std::fabs(S[0][1]), s2 = std::fabs(S[0][2]);
      const double t2 = std::fabs(bvm - S[0][2] * a1 * S[1][2]), t1 = t2 + s1 * gy0, t0 = t1 + s0 * gx0;
      const double e = k1 * bvm + s2 * gze + k1 * s2 * gz0 + u * t2 + s1 * gye + k1 * s1 * gy0 + u * t1 + s0 * gxe + k1 * s0 * gx0 + u * t0;
      fr = std::fmax(fr, e * (1 + 8 * u) / a1);
    }
  }
  std::printf("%.3f %.3f %.3f %.3f %.3f %.3f %.3f\n", (double)log2l(em), (double)log2l(ep), (double)log2l(fm), (double)log2l(ey),
              (double)log2l(fy), std::log2(er), std::log2(fr));
}
"""


def test_bounds_over_the_whole_range(tmp_path):
    nvcc = _build.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", _build.CSRC, "-o", str(exe),
                    str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, check=True, text=True).stdout
    print(out)
    em, ep, fm, ey, fy, er, fr = map(float, out.split())
    # kDfExpRelErr, kE32RelErr; kYRelErr, kY32RelErr; twice those
    assert em <= -31.0 and ep <= -31.0 and fm <= -20.0, out
    assert ey <= -40.0 and fy <= -18.0, out
    assert er <= -39.0 and fr <= -17.0, out
