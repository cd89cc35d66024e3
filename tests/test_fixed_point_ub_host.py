"""The fixed-point sums of the FP64 moment gather without undefined behaviour: compiled
with g++ under its undefined-behaviour checks, on velocities whose positions wrap."""

import os
import shutil
import subprocess

import pytest

from test_fixed_point_host import ROOT

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "fixed_point.cuh"
using namespace fpc;
static double cell(const double *v, int n) {  // [3][n], the mean zero offset U = v's middle
  uint32_t mh[3];
  double U[3];
  for (int d = 0; d < 3; ++d) {
    int32_t lo = 0x7fffffff, hi = -0x7fffffff - 1;
    U[d] = 0;
    for (int i = 0; i < n; ++i) {
      const int32_t k = fx_key((uint32_t)(fx_bits(v[d * n + i]) >> 32));
      lo = k < lo ? k : lo;
      hi = k > hi ? k : hi;
      U[d] += v[d * n + i] / n;
    }
    if (!fx_range(U[d], lo, hi, mh[d])) return -1;
  }
  const FxCell g = fx_cell(mh[0], mh[1], mh[2]);
  FxSums<true> S;
  S.clear(n);
  for (int i = 0; i < n; ++i) {
    if (i == kFxMid) S.carry();
    int64_t c[3];
    for (int d = 0; d < 3; ++d) {
      const int top = g.e[d] + kFxHead + 1023;
      const uint64_t w = fx_bits(v[d * n + i]), u = fx_bits(U[d]);
      c[d] = fx_offset(fx_from_words((uint32_t)(w >> 32), (uint32_t)w, top),
                       fx_from_words((uint32_t)(u >> 32), (uint32_t)u, top));
    }
    fx_accumulate<true>(S, c[0], c[1], c[2], g);
  }
  return std::ldexp((double)fx_fold<true>(S, 0), fx_exponent(fx_weights(0), g)) / n;
}
int main() {
  int taken = 0;
  for (int k = 0; k < 400; ++k) {
    double v[3 * kFxBlock], u11 = 0, m = 0;
    const double at = (k % 2 ? -1 : 1) * std::ldexp(1.0, k % 9);  // means up to 2^8, spreads from 2^2
    for (int i = 0; i < 3 * kFxBlock; ++i) v[i] = at + 4 * std::sin(12.9898 * (i + 1) + k);
    v[0] = at - 4, v[1] = at + 4;
    if (k % 3 == 0) v[2] = -256, v[3] = 256;  // a power of two itself
    for (int i = 0; i < kFxBlock; ++i) m += v[i] / kFxBlock;
    for (int i = 0; i < kFxBlock; ++i) u11 += (v[i] - m) * (v[i] - m) / kFxBlock;
    const double got = cell(v, kFxBlock);
    if (got == -1) continue;
    ++taken;
    if (!(std::fabs(got - u11) <= 1e-13 * u11)) return 1;
  }
  std::printf("%d\n", taken);
  return 0;
}
"""


def test_wrapping_positions(tmp_path):
    """The checks trap on signed overflow and on bad shifts; u_11 of every cell taken is
    right (to 1e-13: some 30 FP64 roundings of the sums it is compared with)."""
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    (tmp_path / "p.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([gxx, "-O1", "-std=c++17", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error", "-I",
                    os.path.join(ROOT, "paper_2606_15622_gb300", "csrc"), str(tmp_path / "p.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0
    assert int(r.stdout) >= 200
