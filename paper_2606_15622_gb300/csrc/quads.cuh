// quads.cuh -- helpers of the kernels that stream particles in quads of four
// consecutive ones (velocity update, adjoint particle pass): vector loads and
// stores of a quad by the alignment class of its component array, and the
// half-warp search of a particle slice's first cell.
#pragma once

#include <cstdint>

namespace fpc {

// Alignment classes of whole quads, per component (bits 2d, 2d + 1): quad Q
// of component d starts at element d np + 4Q - first of two arrays based at
// v and v_out (first: the elements by which particle 0 comes after a quad's
// start)
inline int quad_classes(const void *v, const void *v_out, int64_t np, int64_t first, size_t size) {
  int vec = 0;
  if ((uintptr_t)v % 16 || (uintptr_t)v_out % 16) return 0;
  for (int d = 0; d < 3; ++d) {
    const int e = (int)(((d * np - first % 4) % 4 + 4) % 4);
    const int cls = size == 4 ? (e == 0 ? 2 : (e == 2 ? 1 : 0)) : (e % 2 == 0 ? 2 : 0);
    vec |= cls << (2 * d);
  }
  return vec;
}

// a quad of one component by its alignment class (2: one 16-byte access of
// floats or two of doubles, 1: two 8-byte float pairs, 0: four scalars)
template <typename T>
__device__ __forceinline__ void load_comp(const T *p, int cls, T (&x)[4]);
template <typename T>
__device__ __forceinline__ void store_comp(T *p, int cls, const T (&x)[4]);

// four consecutive values (16-byte aligned address) in and out
__device__ __forceinline__ void load4(const float *p, float (&x)[4]) {
  const float4 a = *reinterpret_cast<const float4 *>(p);
  x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w;
}
__device__ __forceinline__ void load4(const double *p, double (&x)[4]) {
  const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
  x[0] = a.x, x[1] = a.y, x[2] = b.x, x[3] = b.y;
}
__device__ __forceinline__ void store4(float *p, const float (&x)[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void store4(double *p, const double (&x)[4]) {
  reinterpret_cast<double2 *>(p)[0] = make_double2(x[0], x[1]);
  reinterpret_cast<double2 *>(p)[1] = make_double2(x[2], x[3]);
}

template <>
__device__ __forceinline__ void load_comp<float>(const float *p, int cls, float (&x)[4]) {
  if (cls == 2) {
    load4(p, x);
  } else if (cls == 1) {
    const float2 a = reinterpret_cast<const float2 *>(p)[0], b = reinterpret_cast<const float2 *>(p)[1];
    x[0] = a.x, x[1] = a.y, x[2] = b.x, x[3] = b.y;
  } else {
    x[0] = p[0], x[1] = p[1], x[2] = p[2], x[3] = p[3];
  }
}
template <>
__device__ __forceinline__ void load_comp<double>(const double *p, int cls, double (&x)[4]) {
  if (cls == 2)
    load4(p, x);
  else
    x[0] = p[0], x[1] = p[1], x[2] = p[2], x[3] = p[3];
}
template <>
__device__ __forceinline__ void store_comp<float>(float *p, int cls, const float (&x)[4]) {
  if (cls == 2) {
    store4(p, x);
  } else if (cls == 1) {
    reinterpret_cast<float2 *>(p)[0] = make_float2(x[0], x[1]);
    reinterpret_cast<float2 *>(p)[1] = make_float2(x[2], x[3]);
  } else {
    p[0] = x[0], p[1] = x[1], p[2] = x[2], p[3] = x[3];
  }
}
template <>
__device__ __forceinline__ void store_comp<double>(double *p, int cls, const double (&x)[4]) {
  if (cls == 2)
    store4(p, x);
  else
    p[0] = x[0], p[1] = x[1], p[2] = x[2], p[3] = x[3];
}

// FP64 -> T for a table, rounded to nearest even.  To FP32 by integers, which
// does not wait for the FP64 pipe; values beyond FP32's normal range, zeros aside,
// take its conversion.  (That conversion is issued for every value, predicated
// off: the counters show an FP64 instruction a staged word, 14 % of the pipe in
// the particle pass.)
template <typename T>
__device__ __forceinline__ T narrow(double x);
template <>
__device__ __forceinline__ double narrow<double>(double x) { return x; }
template <>
__device__ __forceinline__ float narrow<float>(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  const uint32_t lo = (uint32_t)__double2loint(x);
  const uint32_t a = hi & 0x7fffffffu;
  const bool common = a - (897u << 20) < (253u << 20);  // 2^-126 .. 2^127
  // the top 23 fraction bits under the exponent less 896 (modulo 2^32)
  uint32_t u = __funnelshift_l(lo, hi, 3) - (896u << 23);
  u += ((lo & 0x1fffffffu) + 0x0fffffffu + (u & 1u)) >> 29;
  float f = __uint_as_float((common ? u & 0x7fffffffu : 0u) | (hi & 0x80000000u));
  if (__builtin_expect(!common && (a | lo), 0)) f = (float)x;
  return f;
}

// Rows of NK doubles of up to 32 consecutive cells into shared memory as T,
// row l at stage + l (NK | 1) (an odd stride: the lanes then read their own
// rows without bank conflicts).  The warp's loads are contiguous; a lane that
// read its own row from global memory would touch a line a load (32 wavefronts
// an instruction).
// `more` (if not null): a second set of rows, loaded beside the first into
// stage + more_at.
template <int NK, typename T>
__device__ __forceinline__ void stage_rows(const double *__restrict__ rows, int ncell, T *stage, int lane,
                                           const double *__restrict__ more = nullptr, int more_at = 0) {
  constexpr int kAt = 5;  // loads of a set in flight
  const int total = ncell * NK;
#pragma unroll 1
  for (int t0 = 0; t0 * 32 < total; t0 += kAt) {
    double x[kAt], y[kAt];
#pragma unroll
    for (int t = 0; t < kAt; ++t) {
      const int i = (t0 + t) * 32 + lane;
      if (i < total) {
        x[t] = rows[i];
        if (more) y[t] = more[i];
      }
    }
#pragma unroll
    for (int t = 0; t < kAt; ++t) {
      const int i = (t0 + t) * 32 + lane;
      if (i < total) {
        T *at = stage + i + ((NK | 1) - NK) * (i / NK);
        *at = narrow<T>(x[t]);
        if (more) at[more_at] = narrow<T>(y[t]);
      }
    }
  }
}

// The first cell c in [0, n] with at(c) >= t (at nondecreasing, at(n) >= t),
// found by the 16 lanes of the calling half warp together: each round probes
// 16 evenly spaced cells and keeps the interval where the answer lies, so
// 2^17 cells take five dependent loads.
template <class At>
__device__ __forceinline__ int64_t lower_bound16_by(At at, int64_t n, int64_t t, int lane) {
  const int h = lane & 15;
  const unsigned hmask = 0xffffu << (lane & 16);
  int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (hi - lo > 15) {
    const int64_t step = (hi - lo + 15) / 16;
    const int64_t c = min(lo + step * h, hi);
    const unsigned b = (__ballot_sync(hmask, at(c) >= t) >> (lane & 16)) & 0xffffu;
    if (b == 0) {
      lo = min(lo + step * 15, hi) + 1;
    } else {
      const int f = __ffs(b) - 1;
      if (f == 0) {
        hi = lo;
      } else {
        hi = min(lo + step * f, hi);
        lo = lo + step * (f - 1) + 1;
      }
    }
  }
  const int64_t c = min(lo + h, hi);
  const unsigned b = (__ballot_sync(hmask, at(c) >= t) >> (lane & 16)) & 0xffffu;
  return lo + (__ffs(b) - 1);
}

// the same on the cell offsets: the first cell that starts at or after particle t
__device__ __forceinline__ int64_t lower_bound16(const int64_t *__restrict__ off, int64_t n, int64_t t, int lane) {
  return lower_bound16_by([=](int64_t c) { return off[c]; }, n, t, lane);
}

// Equal shares of a pass over the particles that also prepares every cell: the
// work before particle p of cell c counts as p + kCell (c + 1), before the
// preparation of cell c as off[c] + kCell c.  Share k of n: a warp's particles
// [p0, p1), the cells [c0, c1) whose preparation falls in the share (those
// that it owns), and first = c0 or, where the share starts inside a cell,
// that cell.  (Shares equal in particles alone leave the warps of a rarefied
// region, with ten times the cells, running long after the others.)
struct Share {
  int64_t p0, p1, c0, c1, first;
};
// (n <= 2^14.  Below 2^32 the shares come from 32-bit divisions: a 64-bit one is
// some hundred instructions in a row.)
__device__ __forceinline__ Share warp_share(const int64_t *__restrict__ off, int64_t n_cells, int64_t kCell, uint32_t k,
                                            uint32_t n, int lane) {
  if (n_cells <= 8 * (int64_t)n) {
    // a few whole cells a share: no search (its dependent loads take 3 us);
    // the cells' own offsets bound the particles
    Share s;
    s.c0 = s.first = (int64_t)((uint32_t)n_cells * k / n);
    s.c1 = (int64_t)((uint32_t)n_cells * (k + 1) / n);
    s.p0 = INT64_MIN;
    s.p1 = INT64_MAX;
    return s;
  }
  const int64_t base = off[0], total = off[n_cells] - base + kCell * n_cells;
  const uint32_t kk = lane < 16 ? k : k + 1;
  const int64_t t = base + (total >> 32 == 0 ? (int64_t)((uint32_t)total / n) * kk + (uint32_t)total % n * kk / n
                                             : total / n * kk + total % n * kk / n);
  int64_t c = lower_bound16_by([=](int64_t i) { return off[i] + kCell * i; }, n_cells, t, lane);
  // t lies in cell c - 1: in its preparation (the cell goes to the next share)
  // or among its particles
  int64_t p = off[c];
  if (c > 0) {
    const int64_t q = t - kCell * c;
    if (q <= off[c - 1])
      p = off[--c];
    else if (q < p)
      p = q;
  }
  Share s;
  s.p0 = __shfl_sync(0xffffffffu, p, 0);
  s.p1 = __shfl_sync(0xffffffffu, p, 16);
  s.c0 = __shfl_sync(0xffffffffu, c, 0);
  s.c1 = __shfl_sync(0xffffffffu, c, 16);
  s.first = s.c0 > 0 && off[s.c0] > s.p0 ? s.c0 - 1 : s.c0;
  return s;
}

}  // namespace fpc
