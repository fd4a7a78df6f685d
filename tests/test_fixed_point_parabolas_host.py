"""The FP64 parabolas in fixed point (fix_dev, fix_step4): compiled for the host from the device header and
compared with Sec. 2.1 in 113-bit arithmetic.

Bounds, with u = 2^(E - 1081) the unit of a stencil: a value is cut by less than u, so a difference is off by
at most u, a halved slope by at most 3/2 u (its quarter is cut once more), 3 A by 3 + 2 (3/2 + 3/2) = 9 u and,
where the other edge limits it, by 18 u; the conversion rounds at 2^-53 of the result.  Step 4: num is off by at
most 4 u and s0 by 2 u, so hbar = (20/3) num / s0 - 1 <= 1 by (20/3) 4 u/|s0| + 2 (2 u/|s0|) < 31 u/|s0| (and a few
roundings, 8 2^-52), times |3 h - 3 A| <= 15 |s0| (|A| <= 5 |s0|): 465 u + 120 2^-52 |s0|.  Stencils within 1e-9 of
the one jump of the method, |s0| = min / 100, are left out, and so are ties of its sign tests within 8 u."""
import os
import shutil
import subprocess

import pytest

from test_device_math_host import BEGIN, END, HEADER, PORTABLE, _cuda_include

CODE = r'''
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
#include MHD_DEVICE_HOST_COPY
using namespace mhd;
typedef __float128 Q;
static Q mag(Q x) { return x < 0 ? -x : x; }
static Q half_slope_q(Q a, Q b) {
  if (a * b <= 0) return 0;
  Q m = std::min(std::min(mag(a), mag(b)), mag(a + b) / 4);
  return a < 0 ? -m : m;
}
int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1, 1), E(-40, 40);
  long n = 0, acts = 0, bad = 0, missed = 0, wide = 0, wide_bad = 0, smooth = 0, kept = 0;
  for (long it = 0; it < 1500000; ++it) {
    double q[5];
    const int kind = it % 6;
    const double base = U(g), slope = U(g), curve = U(g), scale = std::exp2(std::floor(E(g)));
    for (int i = 0; i < 5; ++i) {
      const double x = i - 2;
      q[i] = kind == 0 ? U(g)                                            // rough
             : kind == 1 ? 1 + 0.01 * slope * x + 1e-3 * U(g)            // nearly smooth, Step 4 acts
             : kind == 2 ? slope * x + 1e-6 * U(g)                       // through zero
             : kind == 3 ? (x < base * 3 ? 1.0 : 0.02) + 1e-5 * U(g)     // jumps
             : kind == 4 ? base + slope * x + curve * x * x              // parabolas
                         : U(g) * std::exp2(E(g) / 4);                   // many magnitudes
      q[i] *= scale;
    }
    if (it % 101 == 0) q[it % 5] = 0;
    FixCell c[5];
    for (int i = 0; i < 5; ++i) c[i] = fix_cell(q[i]);
    int top = 0;
    for (int i = 0; i < 5; ++i) top = std::max(top, c[i].e);
    Dev<double> P;
    double left;
    FixStep4 st;
    const bool cand = fix_dev(c, P, left, st);
    if (top > std::max(c[2].e, std::min(c[1].e, c[3].e)) + 5) {  // as a whole in FP64
      const Dev<double> W = dev_of(q[0], q[1], q[2], q[3], q[4]);
      ++wide;
      wide_bad += cand || P.A != 3 * W.A || P.B != 3 * W.B || left != q[2] - q[1];
      continue;
    }
    const Q u = std::ldexp(1.0, top - 1081);
    const Q d0 = (Q)q[1] - q[0], d1 = (Q)q[2] - q[1], d2 = (Q)q[3] - q[2], d3 = (Q)q[4] - q[3];
    const Q hm = half_slope_q(d0, d1), h = half_slope_q(d1, d2), hp = half_slope_q(d2, d3);
    Q A = d1 + 2 * (h - hm) / 3, B = d2 - 2 * (hp - h) / 3;
    if (A * B <= 0) A = B = 0;
    else {
      const Q a = A;
      if (mag(A) > 2 * mag(B)) A = 2 * B;
      if (mag(B) > 2 * mag(a)) B = 2 * a;
    }
    const Q Dp = d3 - d2, Dm = d1 - d0, s0 = d1 + d2, mn = std::min(mag(q[1]), mag(q[3]));
    if (mag(mag(s0) - mn / 100) < 1e-9 * mn || (Dp != 0 && mag(Dp) < 8 * u) || (Dm != 0 && mag(Dm) < 8 * u)) continue;
    ++n;
    bad += !(mag(left - d1) <= u + (Q)std::ldexp(1.0, -53) * mag(d1));
    Q hb = 0;
    if (mag(s0) > mn / 100 && Dp * Dm <= 0) {
      hb = (Q)20 / 3 * (Dm - Dp) / s0 - 1;
      hb = hb < 0 ? 0 : hb > 1 ? 1 : hb;
    }
    const Q An = A + hb * (h - A), Bn = B + hb * (h - B);
    const Q tiny = std::ldexp(1.0, -52);
    Q tol = 18 * u;
    if (cand) {
      ++acts;
      P = fix_step4(P, st.num, st.s0, st.h3, fix_min_abs(st), st.E);
      tol += 465 * u + 120 * tiny * mag(s0);
    } else if (hb > 0 && (An != A || Bn != B) && mag(Dm - Dp) > (Q)0.150001 * mag(s0)) {
      ++missed;
    }
    if (!cand) tol += 465 * u * (hb > 0);  // hbar within its error of 0
    bad += !(mag(P.A - 3 * An) <= tol + tiny * mag(3 * An)) || !(mag(P.B - 3 * Bn) <= tol + tiny * mag(3 * Bn));
  }
  for (int i = 0; i < 100000; ++i) {  // a wave resolved by 40 cells
    FixCell c[5];
    for (int j = 0; j < 5; ++j) c[j] = fix_cell(2 + std::sin(2 * M_PI * (i * 0.37 + j) / 40));
    Dev<double> P;
    double left;
    FixStep4 st;
    ++smooth;
    kept += fix_dev(c, P, left, st);
  }
  // infinities and NaNs go the FP64 way; constants give exactly 0, ramps of exact steps exactly their step
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  long special = 0;
  for (int at = 0; at < 5; ++at)
    for (double x : {inf, -inf, nan, 5e306, 1e308, -1.7e308}) {
      double q[5] = {1, 2, 4, 5, 7};
      if (x == 5e306)
        for (double& v : q) v *= 2e306;
      q[at] = x;
      FixCell c[5];
      for (int i = 0; i < 5; ++i) c[i] = fix_cell(q[i]);
      const Dev<double> P = fix_dev_of(c), W = dev_of(q[0], q[1], q[2], q[3], q[4]);
      auto same = [](double a, double b) { return a != a ? b != b : std::fabs(a - b) <= 1e-15 * std::fabs(b) || a == b; };
      special += !same(P.A, W.A) || !same(P.B, W.B);
    }
  for (double x : {0.0, -0.0, 1.0, -3.7e200, 5e-324}) {
    FixCell c[5], r[5];
    for (int i = 0; i < 5; ++i) c[i] = fix_cell(x), r[i] = fix_cell(-1.75 + 0.5 * i);
    Dev<double> P, R;
    double left;
    FixStep4 st;
    special += fix_dev(c, P, left, st) || P.A != 0 || P.B != 0;
    special += fix_dev(r, R, left, st) || R.A != 1.5 || R.B != 1.5;
  }
  std::printf("%ld %ld %ld %ld %ld %ld %ld %ld %ld\n", n, acts, bad, missed, wide, wide_bad, smooth, kept, special);
}
'''


def test_fixed_point_parabolas_match_the_method(tmp_path):
    inc = _cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    src = open(HEADER).read()
    a, b = src.index(BEGIN), src.index(END)
    (tmp_path / "dev.cuh").write_text(src[:a] + PORTABLE + src[b + len(END):])
    (tmp_path / "t.cpp").write_text(CODE)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-w", f"-I{inc}",
                    f'-DMHD_DEVICE_HOST_COPY="{tmp_path / "dev.cuh"}"', str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=300).stdout
    n, acts, bad, missed, wide, wide_bad, smooth, kept, special = (int(x) for x in out.split())
    assert n > 500000 and acts > 50000 and wide > 50000
    assert bad == 0 and missed == 0 and wide_bad == 0 and special == 0
    assert kept < 0.05 * smooth
