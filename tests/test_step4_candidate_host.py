"""The FP64 pencils gather Step 4 of Sec. 2.1 over the warp: a lane hands a parabola on only where
step4_candidate, a test on the high words, says that the blend may act.  Compiled for the host from
the device header: wherever the exact tests hold (D+ D- <= 0, |s0| > mn / 100, hbar > 0) the candidate
test holds, so that leaving the others out changes no bit; and it is not idle (it turns most smooth
stencils down)."""
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
int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(-1, 1), E(-40, 40), near(-2e-6, 2e-6);
  long acts = 0, missed = 0, smooth = 0, kept = 0;
  for (long it = 0; it < 4000000; ++it) {
    const double s0 = U(g) * std::exp2(E(g));
    // num around the threshold 3 |s0| / 20 and mn around 100 |s0|, or anything
    double num = it % 3 == 0 ? s0 * 0.15 * (1 + near(g)) : it % 3 == 1 ? s0 * U(g) : U(g) * std::exp2(E(g));
    double mn = it % 2 == 0 ? std::fabs(s0) * 100 * (1 + near(g)) : std::fabs(U(g)) * std::exp2(E(g));
    if (it % 11 == 0) mn = 0;
    if (it % 13 == 0) num = 0;
    const double Dm = num * (0.5 + 0.5 * std::fabs(U(g))), Dp = it % 17 == 0 ? 0.0 : Dm - num;
    const double n2 = Dm - Dp;
    const Dev<double> P = {U(g), U(g)}, Q = step4(P, 3.0, n2, s0, mn);
    const bool acting = !same_sign(Dp, Dm) && (Q.A != P.A || Q.B != P.B);
    acts += acting;
    missed += acting && !step4_candidate(Dp, Dm, n2, s0, mn);
  }
  for (int i = 0; i < 100000; ++i) {  // a wave resolved by 40 cells
    auto q = [&](int j) { return 2 + std::sin(2 * M_PI * (i * 0.37 + j) / 40); };
    const double Dp = q(2) - 2 * q(1) + q(0), Dm = q(0) - 2 * q(-1) + q(-2);
    ++smooth;
    kept += step4_candidate(Dp, Dm, Dm - Dp, q(1) - q(-1), std::min(q(1), q(-1)));
  }
  std::printf("%ld %ld %ld %ld\n", acts, missed, smooth, kept);
}
'''


def test_no_acting_parabola_is_left_out(tmp_path):
    inc = _cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("needs g++ and the CUDA headers")
    src = open(HEADER).read()
    a, b = src.index(BEGIN), src.index(END)
    (tmp_path / "dev.cuh").write_text(src[:a] + PORTABLE + src[b + len(END):])
    (tmp_path / "t.cpp").write_text(CODE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", f"-I{inc}",
                    f'-DMHD_DEVICE_HOST_COPY="{tmp_path / "dev.cuh"}"', str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=300).stdout
    acts, missed, smooth, kept = (int(x) for x in out.split())
    assert acts > 100000 and missed == 0
    assert kept < 0.05 * smooth
