"""The fixed-point sums of the FP64 moment gather (csrc/fixed_point.cuh, compiled with g++)
over the lanes of its two forms, eight and 32 a cell, on cells whose terms lie close to
their bounds: every integer sum is checked for overflow."""

import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_fixed_point_host import PAIRS, ROOT, TRIPLES, exact

HARNESS = r"""
#include <cmath>
#include "fixed_point.cuh"
using namespace fpc;
// the central sums of one cell by `lanes` lanes, as gather_fp64_kernel forms them; 0: refused,
// -1: an integer sum overflowed
extern "C" int cell(const double *v, int n, const double *U, int lanes, double *out) {
  uint32_t mh[3];
  for (int d = 0; d < 3; ++d) {
    int32_t lo = 0x7fffffff, hi = -0x7fffffff - 1;
    for (int i = 0; i < n; ++i) {
      const int32_t k = fx_key((uint32_t)(fx_bits(v[d * n + i]) >> 32));
      lo = k < lo ? k : lo;
      hi = k > hi ? k : hi;
    }
    if (!fx_range(U[d], lo, hi, mh[d])) return 0;
  }
  const FxCell g = fx_cell(mh[0], mh[1], mh[2]);
  int top[3];
  uint64_t Uf[3];
  for (int d = 0; d < 3; ++d) {
    top[d] = g.e[d] + kFxHead + 1023;
    Uf[d] = (uint64_t)fx_from_words((uint32_t)(fx_bits(U[d]) >> 32), (uint32_t)fx_bits(U[d]), top[d]);
  }
  bool over = false;
  const int fold = fx_fold_bits((n + lanes - 1) / lanes);
  for (int q = 0; q < 26; ++q) out[q] = 0;
  for (int b0 = 0; b0 < n; b0 += lanes * kFxBlock) {
    double block[26] = {};
    for (int l0 = 0; l0 < lanes; l0 += kFxLanes) {
      int64_t f[26] = {};
      for (int l = l0; l < l0 + kFxLanes; ++l) {
        FxSums<true> S;
        int cnt = 0;
        for (int i = b0 + l; i < n && i < b0 + lanes * kFxBlock; i += lanes) ++cnt;
        S.clear(cnt, fold);
        int k = 0;
        for (int i = b0 + l; i < n && i < b0 + lanes * kFxBlock; i += lanes, ++k) {
          if (k == kFxMid) S.carry();
          int64_t c[3];
          for (int d = 0; d < 3; ++d) {
            const uint64_t w = fx_bits(v[d * n + i]);
            c[d] = (int64_t)((uint64_t)fx_from_words((uint32_t)(w >> 32), (uint32_t)w, top[d]) - Uf[d]);
          }
          fx_accumulate<true>(S, c[0], c[1], c[2], g);
        }
        for (int q = 0; q < 26; ++q) over |= __builtin_add_overflow(f[q], fx_fold<true>(S, q, fold), &f[q]);
      }
      for (int q = 0; q < 26; ++q) block[q] += (double)f[q];
    }
    for (int q = 0; q < 26; ++q) out[q] += block[q];
  }
  for (int q = 0; q < 26; ++q) out[q] = std::ldexp(out[q], fx_exponent(fx_weights(q), g, fold));
  return over ? -1 : 1;
}
"""


@pytest.fixture(scope="module")
def cell(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fxl")
    (d / "h.cpp").write_text(HARNESS)
    so = str(d / "h.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2606_15622_gb300", "csrc"), str(d / "h.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).cell
    dp = ctypes.POINTER(ctypes.c_double)

    def call(v, lanes):
        v = np.ascontiguousarray(v, dtype=np.float64)
        U = np.ascontiguousarray(v.sum(axis=1) / v.shape[1])
        out = np.zeros(26)
        ok = fn(v.ctypes.data_as(dp), v.shape[1], U.ctypes.data_as(dp), lanes, out.ctypes.data_as(dp))
        return ok, U, out

    return call


def near_bounds(kind, n, rng):
    """Velocities with many terms near the largest: every component in two cold beams, a
    uniform cube, speeds all alike, beams in x with a plain spread across."""
    if kind == "shell":
        x = rng.standard_normal((3, n))
        return 1.99 * x / np.linalg.norm(x, axis=0)
    if kind == "cube":
        return rng.uniform(-1.95, 1.95, (3, n))
    sign = rng.permutation(np.resize([1.0, -1.0], n))
    v = 0.01 * rng.standard_normal((3, n))
    if kind == "beams across":
        v *= [[1.0], [100.0], [100.0]]
        v[0] += 1.9 * sign
        return v
    return v + {"beams below": 1.95, "beams above": 2.05, "beams low": 1.125}[kind] * sign


@pytest.mark.parametrize("lanes", [8, 32])
@pytest.mark.parametrize("n", [9, 240, 256, 257, 300, 960, 961, 2000])
@pytest.mark.parametrize("kind", ["beams below", "beams above", "beams low", "beams across", "cube", "shell"])
def test_terms_near_their_bounds(cell, kind, n, lanes):
    """2^-48 of the sum of the terms' magnitudes (as for the normal samples; the mean term
    is closer to its bound here)."""
    v = near_bounds(kind, n, np.random.default_rng(n))
    ok, U, got = cell(v, lanes)
    assert ok == 1
    ref, mag = exact(v, U)
    for q in range(26):
        assert abs(Fraction(float(got[q])) - ref[q]) <= mag[q] * Fraction(1, 2**48), q


def fp64_sums(v, U):
    """The 26 sums in FP64 by eight lanes."""
    c = v - U[:, None]
    r2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2]
    rows = ([c[i] * c[j] for i, j in PAIRS] + [c[i] * c[j] * c[k] for i, j, k in TRIPLES]
            + [r2 * (c[i] * c[j]) for i, j in PAIRS] + [r2 * r2 * c[i] for i in range(3)] + [r2 * r2 * r2])
    out = []
    for r in rows:
        lane = np.zeros(8)
        for i in range(0, r.size, 8):
            lane[:r[i:i + 8].size] += r[i:i + 8]
        out.append(((lane[0] + lane[4]) + (lane[2] + lane[6])) + ((lane[1] + lane[5]) + (lane[3] + lane[7])))
    return out


@pytest.mark.parametrize("lanes", [8, 32])
@pytest.mark.parametrize("n", [9, 16, 30, 50, 91])
def test_no_further_off_than_fp64_sums(cell, n, lanes):
    """Over Maxwellian cells and all slots, the root mean square of the errors (in units of
    the sum of the terms' magnitudes) is no larger than that of FP64 sums of the same cells."""
    rng = np.random.default_rng(n)
    fixed, plain = [], []
    for _ in range(30):
        v = rng.standard_normal((3, n)) + np.array([[0.5], [0.0], [-0.2]])
        ok, U, got = cell(v, lanes)
        assert ok == 1
        ref, mag = exact(v, U)
        for errs, x in ((fixed, got), (plain, fp64_sums(v, U))):
            errs.append([float((Fraction(float(x[q])) - ref[q]) / mag[q]) for q in range(26)])
    assert np.sqrt(np.mean(np.square(fixed))) <= np.sqrt(np.mean(np.square(plain)))
