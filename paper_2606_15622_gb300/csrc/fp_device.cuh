// fp_device.cuh -- device helpers shared by the closure kernels (sm_103a).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/fpclosure.h"

namespace fpc {

// ---------------------------------------------------------------------------
// Launches that do not wait for the last kernel's end: launch_after lets the
// kernel's blocks start as the blocks of the stream's kernel before leave the
// SMs; they wait with grid_wait, before their first access to memory, until
// everything that the launch would have waited for is complete and visible.
// The pointers pass through the wait, so that no load through them can be
// moved before it or take the read-only cache, which must not see memory that
// is written while a kernel lives.  Successors may start once every block has
// called grid_wait or grid_release, or ended.
// For chains of short kernels: the sort's eight launches of a collision step
// 504 -> 484 us (131,072 cells) and 153 -> 144 (20,011, LITE), the training
// step's two 57 -> 51.  Not for kernels of few resident blocks an SM (gathers,
// solves, adjoint): blocks that start early crowd on the first SMs that drain
// (exact closure of 131,072 cells 158 -> 207 us, of 16,384 cells 41 -> 47).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename P>
__device__ __forceinline__ void pass_through(P &p) {
  static_assert(sizeof(P) == 8, "a pointer");
  asm volatile("" : "+l"(p)::"memory");
}
template <typename... P>
__device__ __forceinline__ void grid_wait(P &...p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  grid_release();
  (pass_through(p), ...);
}
template <typename... P, typename... A>
inline void launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}


// moment slots (layout documented in fpclosure.h)
constexpr int kN = 0, kU = 1, kTheta = 4, kU2 = 5, kU3 = 11, kW = 21, kZ = 27;
constexpr int kNSum = 26;   // gathered central sums: u2 (6), u3 (10), w (6), z (3), <|c|^6> (1)
constexpr int kNMomSum = 25;  // of those, the ones stored in the moment vector (from slot kU2)
constexpr int kM6Sum = 25;    // the sum slot of <|c|^6> (its own optional output array)

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): the counter-based
// generator of the noise variates and of the dropout masks.  The key
// schedule (k0 + r 0x9E3779B9, k1 + r 0xBB67AE85 for round r) depends on the
// seed only, so the host computes it once (philox_keys) and passes it as a
// kernel parameter.
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};

__device__ __forceinline__ uint4 philox4x32_10(uint4 x, const PhiloxKeys &key) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // one 32x32 -> 64-bit multiply gives both halves of each product
    const uint64_t p0 = (uint64_t)0xD2511F53u * x.x, p1 = (uint64_t)0xCD9E8D57u * x.z;
    x = make_uint4((uint32_t)(p1 >> 32) ^ x.y ^ key.k0[r], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ x.w ^ key.k1[r],
                   (uint32_t)p0);
  }
  return x;
}

inline PhiloxKeys philox_keys(uint64_t seed) {
  PhiloxKeys k;
  for (int r = 0; r < 10; ++r) {
    k.k0[r] = (uint32_t)seed + 0x9E3779B9u * (uint32_t)r;
    k.k1[r] = (uint32_t)(seed >> 32) + 0xBB67AE85u * (uint32_t)r;
  }
  return k;
}

// Conversions between binary64 and binary32 done with integer operations on
// the IEEE-754 bit layouts.  On this chip the FP64 pipe executes conversion
// instructions too, and it is the scarcest pipe; these keep per-cell
// bookkeeping off it.
//   f2d_exact:  float -> double, exact (below);
//   d2f_rn:     double -> float rounded to nearest, ties to even; results
//               below the smallest normal float are flushed to a signed zero,
//               beyond the largest give infinity, NaN stays NaN;
//   u2d_exact:  32-bit unsigned integer -> double, exact.
__device__ __forceinline__ float d2f_rn(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  if (e == 0x7ff) return __uint_as_float(sign | 0x7f800000u | (((hi & 0xfffffu) | lo) ? 0x400000u : 0u));
  const int eb = e - 896;  // biased binary32 exponent
  if (eb >= 255) return __uint_as_float(sign | 0x7f800000u);
  if (eb <= 0) return __uint_as_float(sign);
  const uint32_t m = ((hi & 0xfffffu) << 3) | (lo >> 29);  // the top 23 of the 52 fraction bits
  const uint32_t rest = lo & 0x1fffffffu;                   // the 29 bits below them
  const uint32_t up = (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
  // a carry out of the fraction moves into the exponent (and to infinity at the top)
  return __uint_as_float(sign | ((((uint32_t)eb << 23) | m) + up));
}

__device__ __forceinline__ double u2d_exact(uint32_t n) {
  if (n == 0u) return 0.0;
  const int e = 31 - __clz(n);                                             // 2^e <= n < 2^(e+1)
  const uint64_t frac = ((uint64_t)n << (52 - e)) & 0xfffffffffffffull;  // drop the leading one
  return __longlong_as_double((long long)(((uint64_t)(e + 1023) << 52) | frac));
}

// |x| as its bits, put together from the halves: masked as one 64-bit word the
// compiler sees an absolute value and takes it, and the comparisons, to the
// FP64 pipe
__device__ __forceinline__ uint64_t abs_bits(double x) {
  uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  asm("" : "+r"(hi));
  return ((uint64_t)hi << 32) | (uint32_t)__double2loint(x);
}
__device__ __forceinline__ bool finite_d(double x) {
  return (abs_bits(x) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}

// x 2^k exactly on the integer pipe: the exponent's field raised, a subnormal
// shifted (its leading bit moves into the exponent), an overflow to infinity,
// infinities and NaN as they are.
template <int k>
__host__ __device__ __forceinline__ double times_pow2(double x) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t a = hi & 0x7fffffffu;
  uint32_t h = hi + ((uint32_t)k << 20), l = lo;
  if (__builtin_expect(a - (1u << 20) >= (uint32_t)(2046 - k) << 20, 0)) {
    asm volatile("" : "+r"(l));  // a branch, not computed beside the common case
    uint64_t b = ((uint64_t)a << 32) | lo;
#pragma unroll
    for (int i = 0; i < k; ++i) {
      if (b < (1ull << 52))
        b <<= 1;
      else if (b < (2047ull << 52))
        b = b >= (2046ull << 52) ? 2047ull << 52 : b + (1ull << 52);
    }
    h = (uint32_t)(b >> 32) | (hi & 0x80000000u);
    l = (uint32_t)b;
  }
  return __hiloint2double((int)h, (int)l);
#else
  return x * (double)(1 << k);
#endif
}

// 1 / p from the hardware's FP32 reciprocal of p's mantissa (good to about
// 2^-22) and one step of third order on it, x (1 + e + e^2) with e = 1 - m x:
// what is left out, e^3, is below 2^-64, so the result is within a little over
// half a unit in the last place (a subnormal one is cut off).  The exponent and
// the special values are put in by integer operations: three FP64 instructions
// where the division takes about ten.
__host__ __device__ __forceinline__ double rcp_d(double p) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)__double2hiint(p), sign = hi & 0x80000000u;
  uint32_t mh = hi & 0x000fffffu, ml = (uint32_t)__double2loint(p);  // the fraction
  int ex = (int)((hi >> 20) & 0x7ffu);
  if (__builtin_expect(ex == 0, 0)) {  // subnormal: the leading bit to the place before the fraction
    asm volatile("" : "+r"(mh));       // (a branch, as below)
    const uint64_t f = ((uint64_t)mh << 32) | ml;
    const int sh = f ? __clzll((long long)f) - 11 : 0;
    mh = (uint32_t)((f << sh) >> 32) & 0x000fffffu;
    ml = (uint32_t)(f << sh);
    ex = f ? 1 - sh : -2000;  // (zero: infinity below)
  }
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | __funnelshift_l(ml, mh, 3))));
  const uint32_t rb = __float_as_uint(r);  // in [1/2, 1]
  const double m = __hiloint2double((int)(mh | 0x3ff00000u), (int)ml);
  double x = __hiloint2double((int)((rb >> 3) + (896u << 20)), (int)(rb << 29));
  double e = fma(-m, x, 1.0);
  e = fma(e, e, e);
  x = fma(x, e, x);
  const uint32_t xh = (uint32_t)__double2hiint(x);
  uint32_t oh = xh + ((uint32_t)(1023 - ex) << 20), ol = (uint32_t)__double2loint(x);
  if (__builtin_expect((unsigned)(ex - 1) >= 2044u, 0)) {
    asm volatile("" : "+r"(ol));
    const int oe = (int)(xh >> 20) + 1023 - ex;  // the result's exponent field
    if (ex == 0x7ff) {
      oh = (mh | ml) ? 0x7ff80000u : 0u;
      ol = 0u;
    } else if (oe >= 2047) {
      oh = 0x7ff00000u;
      ol = 0u;
    } else if (oe <= 0) {  // subnormal, by one or two bits
      const uint32_t g = (xh & 0x000fffffu) | 0x00100000u;
      ol = __funnelshift_r(ol, g, 1 - oe);
      oh = g >> (1 - oe);
    }
  }
  return __hiloint2double((int)(oh | sign), (int)ol);
#else
  return 1.0 / p;
#endif
}

// x > 0 for a double (false for NaN), on its bits
__device__ __forceinline__ bool positive_d(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}

// Error-free transformation a + b = s + e (Knuth two-sum).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// Order of the central moment held in gathered sum slot q (0..25).
__host__ __device__ constexpr int sum_order(int q) {
  return q < 6 ? 2 : (q < 16 ? 3 : (q < 22 ? 4 : (q < 25 ? 5 : 6)));
}

// Butterfly all-reduce over groups of G consecutive lanes (all 32 lanes call).
template <int G, typename T>
__device__ __forceinline__ T group_allreduce(T x) {
#pragma unroll
  for (int o = G / 2; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Reduce-scatter of 32 slots over groups of G lanes: on return lane l of the
// group holds, in hi / lo[0 .. 32/G), the group sums of slots [l*32/G,
// (l+1)*32/G), as compensated pairs: hi sums by two-sum, errors and lo parts
// accumulated in lo.
template <int G>
__device__ __forceinline__ void group_reduce_scatter2(float (&hi)[32], float (&lo)[32], int lane) {
#pragma unroll
  for (int lvl = 0; (G >> (lvl + 1)) >= 1; ++lvl) {
    const int o = G >> (lvl + 1);
    const int half = 16 >> lvl;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      float sh = up ? hi[j] : hi[j + half];
      float sl = up ? lo[j] : lo[j + half];
      float kh = up ? hi[j + half] : hi[j];
      float kl = up ? lo[j + half] : lo[j];
      float rh = __shfl_xor_sync(0xffffffffu, sh, o);
      float rl = __shfl_xor_sync(0xffffffffu, sl, o);
      float s, e;
      two_sum(kh, rh, s, e);
      hi[j] = s;
      lo[j] = (kl + rl) + e;
    }
  }
}

template <typename VT>
__device__ __forceinline__ VT ldg_v(const VT *p) { return __ldg(p); }

// Exact float -> double by integer bit manipulation (no FP64-pipe work), with
// an optional power-of-two scale 2^exp_add folded into the exponent.
// Normal floats and zeros convert exactly; FP32 subnormals flush to zero;
// results outside the double range saturate to zero / infinity; inf and NaN
// pass through.
__device__ __forceinline__ double f2d_exact(float f, int exp_add = 0) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t sign = u & 0x80000000u;
  const int e = (int)((u >> 23) & 0xffu);
  const uint32_t man = u & 0x7fffffu;
  const int ed = e + (1023 - 127) + exp_add;
  uint32_t hi = sign | (man >> 3), lo = man << 29;
  if (e == 0 || ed <= 0) {
    hi = sign;
    lo = 0u;
  } else if (e == 255 || ed >= 2047) {
    hi |= 0x7ff00000u;
    if (e != 255) {
      hi = sign | 0x7ff00000u;
      lo = 0u;
    }
  } else {
    hi |= (uint32_t)ed << 20;
  }
  return __hiloint2double((int)hi, (int)lo);
}

// Double-float helpers (pairs of FP32 carrying ~46 significant bits).
// (rh, rl) ~ 1/n: rh the rounded reciprocal, rl its residual.
__device__ __forceinline__ void df_recip(float n, float &rh, float &rl) {
  rh = __frcp_rn(n);
  rl = fmaf(-rh, n, 1.f) * rh;
}
// (hi + lo) * (rh + rl) as a double-float (p, e)
__device__ __forceinline__ void df_scale(float hi, float lo, float rh, float rl, float &p, float &e) {
  p = hi * rh;
  e = fmaf(hi, rh, -p);
  e = fmaf(hi, rl, fmaf(lo, rh, e));
}

// Copy a per-cell constant row (NC entries, 16-byte aligned, NC a multiple of
// four) from shared memory into registers with 16-byte loads.
template <int NC>
__device__ __forceinline__ void load_row(const float *__restrict__ row, float (&K)[NC]) {
  static_assert(NC % 4 == 0, "row length");
  const float4 *r4 = reinterpret_cast<const float4 *>(row);
#pragma unroll
  for (int q = 0; q < NC / 4; ++q) {
    const float4 x = r4[q];
    K[4 * q] = x.x;
    K[4 * q + 1] = x.y;
    K[4 * q + 2] = x.z;
    K[4 * q + 3] = x.w;
  }
}
template <int NC>
__device__ __forceinline__ void load_row(const double *__restrict__ row, double (&K)[NC]) {
  static_assert(NC % 2 == 0, "row length");
  const double2 *r2 = reinterpret_cast<const double2 *>(row);
#pragma unroll
  for (int q = 0; q < NC / 2; ++q) {
    const double2 x = r2[q];
    K[2 * q] = x.x;
    K[2 * q + 1] = x.y;
  }
}

// and back
template <int NC>
__device__ __forceinline__ void store_row(float *row, const float (&K)[NC]) {
  static_assert(NC % 4 == 0, "row length");
#pragma unroll
  for (int q = 0; q < NC / 4; ++q)
    reinterpret_cast<float4 *>(row)[q] = make_float4(K[4 * q], K[4 * q + 1], K[4 * q + 2], K[4 * q + 3]);
}
template <int NC>
__device__ __forceinline__ void store_row(double *row, const double (&K)[NC]) {
  static_assert(NC % 2 == 0, "row length");
#pragma unroll
  for (int q = 0; q < NC / 2; ++q) reinterpret_cast<double2 *>(row)[q] = make_double2(K[2 * q], K[2 * q + 1]);
}

}  // namespace fpc
