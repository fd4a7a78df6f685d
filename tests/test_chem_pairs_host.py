"""The H/H2 network of the FP32-bulk path in pairs of floats (chem_cell_pairs), compiled for the host from
the device header, against the FP64 evaluation of the same cell (chem_cell): the stored 24-bit rho_H2 is the
FP64 result rounded once.  A pair evaluation good to 2^-40 of the densities involved can differ from
that only next to a rounding boundary, so every case is within half an ulp and 2^-14 of an ulp of
the FP64 value; the share of cells whose stored bits differ is then about 2^-15.  Cold to hot gas, thin to dense,
atomic to molecular, at equilibrium, short to long steps, several shielding lengths; inputs outside
the pairs' range (zero, negative, huge, NaN) are handed back to FP64."""
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
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(0, 1);
  long n = 0, off = 0, differ = 0, handed = 0;
  double worst = 0;
  for (long it = 0; it < 1000000; ++it) {
    Phys ph{};
    ph.chem = 1;
    ph.dx = std::pow(10.0, -2 + 4 * U(g));
    ph.bdop = 0.5 + 5 * U(g);
    ph.xnorm = 5e14 * std::pow(10.0, 2 * U(g) - 1);
    ph.taud = it % 3 ? 1e-21 : 1e-22 * U(g);
    ph.ibdop = 1 / ph.bdop;
    ph.ixnorm = 1 / ph.xnorm;
    set_shielding(ph);
    const float rho = (float)std::pow(10.0, -3 + 7 * U(g));
    const double f = it % 4 == 0 ? 0.0 : it % 4 == 1 ? 1.0 - 1e-3 * U(g) : U(g);
    float rh2 = (float)(rho * f);
    const double T = std::pow(10.0, 0.5 + 5 * U(g)), n1 = rho - rh2, n2 = 0.5 * rh2;
    const float e = (float)((3 * n1 + 5 * n2) * 0.5 * T * ChemConst::KB / (ChemConst::MH * 1e10));
    const double tau = std::pow(10.0, -4 + 4 * U(g)), tss = tau * (ChemConst::PC / ChemConst::KMS);
    const float ts[2] = {(float)tss, (float)(tss - (double)(float)tss)};
    if (it % 7 == 0 && f > 0) {  // near equilibrium: a long step from there
      const ChemOut q = chem_cell<false>(ph, rho, e, rh2, 0.0, 1e3 * tau);
      rh2 = (float)q.rh2;
    }
    const ChemOut want = chem_cell<false>(ph, rho, e, rh2, 0.0, tau);
    float got;
    if (!chem_cell_pairs(ph, ts, rho, e, rh2, got)) { ++handed; continue; }
    ++n;
    if (want.rh2 < 1e-30) { off += std::fabs((double)got - want.rh2) > 1e-30; continue; }
    const double ulp = std::ldexp(1.0, std::ilogb(want.rh2) - 23);
    const double err = std::fabs((double)got - want.rh2) / ulp;
    worst = std::max(worst, err);
    off += err > 0.5 + std::ldexp(1.0, -14);
    differ += got != (float)want.rh2;
  }
  Phys ph{};
  ph.dx = 1; ph.bdop = 3; ph.ibdop = 1 / 3.0; ph.xnorm = 5e14; ph.ixnorm = 2e-15; ph.taud = 1e-21;
  set_shielding(ph);
  const float ts[2] = {1e12f, 0.f}, nan = std::numeric_limits<float>::quiet_NaN(), inf = std::numeric_limits<float>::infinity();
  const float bad[][3] = {{0, 1, 0}, {-1, 1, 0}, {1, 0, 0}, {1, -1, 0}, {1, 1, -1}, {nan, 1, 0}, {1, nan, 0}, {1, 1, nan},
                          {inf, 1, 0}, {1, inf, 0}, {1, 1, inf}, {1e30f, 1, 0}, {1, 1e30f, 0}, {1, 1, 2.5f}};
  long taken = 0;
  for (auto& b : bad) { float r; taken += chem_cell_pairs(ph, ts, b[0], b[1], b[2], r); }
  std::printf("%ld %ld %ld %ld %ld %.6f\n", n, off, differ, handed, taken, worst);
}
'''


def test_pairs_store_the_fp64_result(tmp_path):
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
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=300).stdout.split()
    n, off, differ, handed, taken = (int(x) for x in out[:5])
    assert n > 900000, out
    assert off == 0, out
    assert differ <= 2 ** -13 * n, out
    assert taken == 0, out
