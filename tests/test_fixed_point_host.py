"""The fixed-point sums of the FP64 moment gather (csrc/fixed_point.cuh, compiled
with g++) against exact rational sums: every cell that the form takes, over
spreads, offsets, thin distributions and sizes, and the cells that it refuses."""

import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cmath>
#include "fixed_point.cuh"
using namespace fpc;
// the central sums of one cell, eight lanes, as gather_fp64_kernel forms them; 0: refused
extern "C" int cell(const double *v, int n, const double *U, double *out) {
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
  int64_t Uf[3];
  for (int d = 0; d < 3; ++d) {
    top[d] = g.e[d] + kFxHead + 1023;
    Uf[d] = fx_from_words((uint32_t)(fx_bits(U[d]) >> 32), (uint32_t)fx_bits(U[d]), top[d]);
  }
  for (int q = 0; q < 26; ++q) out[q] = 0;
  for (int b0 = 0; b0 < n; b0 += 8 * kFxBlock) {
    int64_t f[26] = {};
    for (int l = 0; l < 8; ++l) {
      FxSums<true> S;
      int cnt = 0;
      for (int i = b0 + l; i < n && i < b0 + 8 * kFxBlock; i += 8) ++cnt;
      S.clear(cnt);
      int k = 0;
      for (int i = b0 + l; i < n && i < b0 + 8 * kFxBlock; i += 8, ++k) {
        if (k == kFxMid) S.carry();
        int64_t c[3];
        for (int d = 0; d < 3; ++d) {
          const uint64_t w = fx_bits(v[d * n + i]);
          c[d] = (int64_t)((uint64_t)fx_from_words((uint32_t)(w >> 32), (uint32_t)w, top[d]) - (uint64_t)Uf[d]);
        }
        fx_accumulate<true>(S, c[0], c[1], c[2], g);
      }
      for (int q = 0; q < 26; ++q) f[q] += fx_fold<true>(S, q);
    }
    for (int q = 0; q < 26; ++q) out[q] += (double)f[q];
  }
  for (int q = 0; q < 26; ++q) out[q] = std::ldexp(out[q], fx_exponent(fx_weights(q), g));
  return 1;
}
"""

PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
TRIPLES = [(0, 0, 0), (0, 0, 1), (0, 0, 2), (0, 1, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2),
           (2, 2, 2)]


@pytest.fixture(scope="module")
def cell(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("fx")
    (d / "h.cpp").write_text(HARNESS)
    so = str(d / "h.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2606_15622_gb300", "csrc"), str(d / "h.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).cell
    dp = ctypes.POINTER(ctypes.c_double)

    def call(v):
        v = np.ascontiguousarray(v, dtype=np.float64)
        with np.errstate(all="ignore"):
            U = np.ascontiguousarray(v.sum(axis=1) / v.shape[1])
        out = np.zeros(26)
        ok = fn(v.ctypes.data_as(dp), v.shape[1], U.ctypes.data_as(dp), out.ctypes.data_as(dp))
        return bool(ok), U, out

    return call


def exact(v, U):
    """The 26 sums about U as rationals, and the sums of the terms' magnitudes."""
    c = [[Fraction(float(x)) - Fraction(float(U[d])) for x in v[d]] for d in range(3)]
    rows = []
    for x in zip(*c):
        r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2]
        rows.append([x[i] * x[j] for i, j in PAIRS] + [x[i] * x[j] * x[k] for i, j, k in TRIPLES]
                    + [r2 * x[i] * x[j] for i, j in PAIRS] + [r2 * r2 * x[i] for i in range(3)] + [r2 * r2 * r2])
    return [sum(col) for col in zip(*rows)], [sum(abs(y) for y in col) for col in zip(*rows)]


@pytest.mark.parametrize("n", [2, 8, 9, 91, 256, 257, 2000])
@pytest.mark.parametrize("U,sigma", [((0, 0, 0), (1, 1, 1)), ((12.9, 0, -3), (1, 1, 1)),
                                     ((0, 0, 0), (1, 30, 1e-3)), ((1e-20, 0, 0), (1e-20, 3e-20, 1e-21)),
                                     ((-5e12, 0, 0), (1e12, 1e13, 2e12))])
def test_sums_against_rationals(cell, n, U, sigma):
    """Each error at most 2^-48 of the sum of the terms' magnitudes: a term's error is
    a few units of 2^-58 of the largest possible term, which for these samples (|c|
    up to about 2^3 sigma once its bound is a power of two) is below 2^9 of the mean
    term of the highest order."""
    rng = np.random.default_rng(n)
    v = np.array(U, float)[:, None] + np.array(sigma, float)[:, None] * rng.standard_normal((3, n))
    ok, Um, got = cell(v)
    assert ok
    ref, mag = exact(v, Um)
    for q in range(26):
        assert abs(Fraction(float(got[q])) - ref[q]) <= mag[q] * Fraction(1, 2**48), q


def test_offset_beyond_a_word_wraps_exactly(cell):
    """64 times the spread from zero, the largest offset taken: differences are exact
    although the fixed-point positions wrap."""
    rng = np.random.default_rng(5)
    v = 100.0 + rng.uniform(-1.55, 1.55, (3, 40))
    v[:, 0], v[:, 1] = 98.45, 101.55
    ok, Um, got = cell(v)
    assert ok
    ref, mag = exact(v, Um)
    assert all(abs(Fraction(float(got[q])) - ref[q]) <= mag[q] * Fraction(1, 2**48) for q in range(26))


@pytest.mark.parametrize("bad", ["nan", "inf", "alike", "cold", "tiny", "huge"])
def test_refused_cells(cell, bad):
    rng = np.random.default_rng(7)
    v = rng.standard_normal((3, 20))
    if bad in ("nan", "inf"):
        v[1, 3] = float(bad)
    elif bad == "alike":
        v[2] = 0.75
    elif bad == "cold":
        v[0] = 1000.0 + v[0]
    else:
        v *= 1e-40 if bad == "tiny" else 1e40
    assert not cell(v)[0]
