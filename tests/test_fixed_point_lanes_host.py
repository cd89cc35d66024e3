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
// 2: its tails are too heavy, -1: an integer sum overflowed
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
  const int u[3] = {0, 3, 5};
  const auto hi = [](double x) { return (uint32_t)(fx_bits(x) >> 32); };
  int32_t lmax = 0;
  for (int d = 0; d < 3; ++d) {
    const int32_t lu = fx_log(hi(out[u[d]]), g.e[d], fold);
    lmax = lu > lmax ? lu : lmax;
  }
  bool heavy = false;
  for (int d = 0; d < 3; ++d) heavy |= fx_heavy(hi(out[16 + u[d]]), hi(out[u[d]]), hi(n), g.er, lmax);
  for (int q = 0; q < 26; ++q) out[q] = std::ldexp(out[q], fx_exponent(fx_weights(q), g, fold));
  if (heavy) return 2;
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


def heavy(kind, n, rng):
    """Maxwellian cells with outliers in one or two components, hot tails, Student's t."""
    v = rng.standard_normal((3, n))
    if kind == "student":
        return rng.standard_t(3, (3, n))
    if kind == "hot tail":
        v[:, rng.random(n) < 0.02] *= 6.5
    else:
        size, components = kind
        for d in range(components):
            v[d, d] = size * (1 + 0.1 * rng.random())
    return v


HEAVY = ["student", "hot tail"] + [(size, k) for size in (6, 10, 30, 1e3, 1e6) for k in (1, 2)]


def bounds(mag, most, n):
    """What a cell's sums may be off by: FP64 sums by eight lanes add n / 8 terms a lane and
    round terms and lanes' sums some 16 times, 2^-53 of the terms' magnitudes `mag` each.
    Cells of up to 16 particles are never taken for heavy, so there also the fixed-point
    form's own part: up to 8 units of 2^-58 of the largest possible term a particle, whose
    factors are bounded by powers of two (|c_d| < 2 max |c_d|, |c|^2 < 8 sum max c_d^2)."""
    m = [2 * x for x in most]
    r2 = 2 * sum(x * x for x in m)
    top = ([m[i] * m[j] for i, j in PAIRS] + [m[i] * m[j] * m[k] for i, j, k in TRIPLES]
           + [r2 * m[i] * m[j] for i, j in PAIRS] + [r2 * r2 * m[i] for i in range(3)] + [r2 * r2 * r2])
    return [a * (n // 8 + 16) * 2.0**-53 + (n * t * 2.0**-55 if n <= 16 else 0.0) for a, t in zip(mag, top)]


@pytest.mark.parametrize("lanes", [8, 32])
@pytest.mark.parametrize("kind", HEAVY, ids=str)
def test_heavy_tails(cell, kind, lanes):
    """Cells that fixed point takes stay within `bounds`."""
    rng = np.random.default_rng(1)
    for n in (9, 16, 30, 100, 300, 1000):
        v = heavy(kind, n, rng)
        ok, U, got = cell(v, lanes)
        assert ok in (1, 2)
        if ok == 1:
            ref, mag = exact(v, U)
            for q, most in enumerate(bounds([float(x) for x in mag], np.abs(v - U[:, None]).max(1), n)):
                assert abs(Fraction(float(got[q])) - ref[q]) <= most, (n, q)


def test_maxwellian_cells_are_taken(cell):
    rng = np.random.default_rng(2)
    for n in (9, 12, 20, 50, 200):
        for _ in range(200):
            assert cell(rng.standard_normal((3, n)) * [[1.0], [2.0], [0.5]], 8)[0] == 1
