// gather_fp64.cu -- FP64 moment gather (paper Sec. 3.6 moments) for sm_103a.
//
// Eight lanes a cell, four cells of similar size a warp task (small problems:
// a warp a cell), two passes over the cell's particles:
//   pass A  the FP64 sum of the velocities (U) and, on the integer pipe, the
//           least and largest high word of every component, which bound
//           |v - U|;
//   pass B  c = v - U and the 26 central sums in 58-bit fixed point
//           (fixed_point.cuh), folded over the group's lanes by a shared-memory
//           transpose into FP64.
// The first pass streams the velocities from DRAM, the second re-reads them
// from L1 / L2.  What bounds it: instruction issue on the integer pipes, whose
// 32 x 32-bit wide products (74 a particle) issue every 4 to 6 cycles; the
// same sums on the FP64 pipe take 41 instructions of 68 cycles each.  On
// 131,072 cells of 11.9M particles: 0.41 ms, where FP64 sums took 1.75 ms (and
// still do where every cell takes them).
// Every warp of a resident grid takes an equal share of the work and walks its
// cells in runs of up to 32, ranked by size so that the four cells of a task
// have similar trip counts.
//
// A cell outside the fixed-point form's reach takes its sums in FP64: a
// velocity that is not finite, a component whose spread is below 2^-5 of its
// speed or that does not vary at all, a spread beyond 2^+-120 (FP32 velocities:
// below 2^-67), tails so heavy that fixed point loses digits (fx_heavy; known
// after the sums), and cells of up to eight particles (one round of the lanes; their systems can be so
// ill-conditioned that every rounding shows).
#include <cstdint>

#include "fixed_point.cuh"
#include "fp_device.cuh"
#include "quads.cuh"

namespace fpc {

constexpr int kGWarps = 4;           // warps per block
constexpr int kGAhead = 4;           // particles a lane loads ahead in pass A
constexpr int kGBlocksPerSm = 3;
constexpr int kGFew = 8;             // cells of up to so many particles in FP64
constexpr int64_t kGCellWork = 28;   // a cell's fixed work in particles (instructions a task / a particle)

__device__ __forceinline__ void accumulate26d(double (&t)[kNSum], double cx, double cy, double cz) {
  const double xx = cx * cx, xy = cx * cy, xz = cx * cz, yy = cy * cy, yz = cy * cz, zz = cz * cz;
  t[0] += xx; t[1] += xy; t[2] += xz; t[3] += yy; t[4] += yz; t[5] += zz;
  t[6] = fma(xx, cx, t[6]);  t[7] = fma(xx, cy, t[7]);   t[8] = fma(xx, cz, t[8]);
  t[9] = fma(xy, cy, t[9]);  t[10] = fma(xy, cz, t[10]); t[11] = fma(xz, cz, t[11]);
  t[12] = fma(yy, cy, t[12]); t[13] = fma(yy, cz, t[13]); t[14] = fma(yz, cz, t[14]);
  t[15] = fma(zz, cz, t[15]);
  const double r2 = xx + yy + zz;
  t[16] = fma(r2, xx, t[16]); t[17] = fma(r2, xy, t[17]); t[18] = fma(r2, xz, t[18]);
  t[19] = fma(r2, yy, t[19]); t[20] = fma(r2, yz, t[20]); t[21] = fma(r2, zz, t[21]);
  const double r4 = r2 * r2;
  t[22] = fma(r4, cx, t[22]); t[23] = fma(r4, cy, t[23]); t[24] = fma(r4, cz, t[24]);
  t[25] = fma(r4, r2, t[25]);
}

// a velocity as the two words of its double (FP32 values on the integer pipe;
// FP32 subnormals read as zero there: see kFxMinExpF)
__device__ __forceinline__ uint2 v_words(double x) {
  return make_uint2((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x));
}
__device__ __forceinline__ uint2 v_words(float x) {
  const double d = f2d_exact(x);
  return make_uint2((uint32_t)__double2hiint(d), (uint32_t)__double2loint(d));
}

// 1 / n to the last bit: an FP32 reciprocal and two Newton steps
__device__ __forceinline__ double recip_count(int n) {
  const double d = u2d_exact((uint32_t)n);
  double y = f2d_exact(__frcp_rn((float)n));
  y = fma(y, fma(-d, y, 1.0), y);
  return fma(y, fma(-d, y, 1.0), y);
}

// reduce-scatter of three values over the G lanes of a group: lane lg gets
// component lg & 3 (3: pad).  Lanes 4 and more apart are added first.
template <int G, typename T, class Op>
__device__ __forceinline__ T group_scatter3(T a, T b, T c, T pad, int lg, Op op) {
#pragma unroll
  for (int o = G / 2; o >= 4; o >>= 1) {
    a = op(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = op(b, __shfl_xor_sync(0xffffffffu, b, o));
    c = op(c, __shfl_xor_sync(0xffffffffu, c, o));
  }
  const bool hi = (lg & 2) != 0;
  T k0 = hi ? c : a, k1 = hi ? pad : b;
  k0 = op(k0, __shfl_xor_sync(0xffffffffu, hi ? a : c, 2));
  k1 = op(k1, __shfl_xor_sync(0xffffffffu, hi ? b : pad, 2));
  const bool od = (lg & 1) != 0;
  T k = od ? k1 : k0;
  return op(k, __shfl_xor_sync(0xffffffffu, od ? k0 : k1, 1));
}

// the slots that lane lg of a group owns after group_transpose: the pairs
// 2 (lg & 7) of each half of 16
constexpr int kOwn = 4;
__device__ __forceinline__ int own_slot(int k, int lg) { return 16 * (k >> 1) + 2 * (lg & 7) + (k & 1); }

// The 26 slots of the group's G lanes summed, each by the lanes that own it
// (G = 32: four lanes): eight lanes' in T, the eights in FP64 (integer sums
// have room for kFxLanes lanes).  get(q) is the lane's own slot q (q a
// constant after unrolling).  sc: the warp's scratch (32 rows of 128 bytes, the
// chunks of a row rotated so that a quarter-warp's 16-byte accesses hit all
// banks).
template <int G, typename T, class Get>
__device__ __forceinline__ void group_transpose(Get get, double (&out)[kOwn], T *sc, int lane) {
  static_assert(sizeof(T) == 8, "two slots a 16-byte chunk");
  struct alignas(16) Two {
    T a, b;
  };
  constexpr int kRows = 8;  // rows a lane adds
  static_assert(kRows == kFxLanes, "integer sums of so many lanes");
  Two *s2 = reinterpret_cast<Two *>(sc);
  const int ch = lane & 7, base = lane & ~7;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const int q = 16 * half + 2 * w;
      if (q < kNSum) s2[lane * 8 + (w ^ ch)] = Two{get(q), get(q + 1)};
    }
    __syncwarp();
    double a = 0.0, b = 0.0;
    if (16 * half + 2 * ch < kNSum) {
      T ra[kRows], rb[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        const Two t = s2[(base + i) * 8 + (ch ^ i)];
        ra[i] = t.a;
        rb[i] = t.b;
      }
#pragma unroll
      for (int o = kRows / 2; o >= 1; o >>= 1)  // rows far apart first
#pragma unroll
        for (int i = 0; i < o; ++i) {
          ra[i] += ra[i + o];
          rb[i] += rb[i + o];
        }
      a = (double)ra[0];
      b = (double)rb[0];
    }
#pragma unroll
    for (int o = 8; o < G; o <<= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    out[2 * half] = a;
    out[2 * half + 1] = b;
    __syncwarp();
  }
}

template <typename VT, bool kM6, int G>
__global__ void __launch_bounds__(32 * kGWarps, kGBlocksPerSm)
    gather_fp64_kernel(const VT *__restrict__ v, int64_t np, const int64_t *__restrict__ off, int64_t n_cells,
                       double *__restrict__ mom, double *__restrict__ m6) {
  __shared__ __align__(16) int64_t scratch[kGWarps][32 * 16];
  const int lane = threadIdx.x & 31;
  constexpr int kCells = 32 / G;  // a task
  const int lg = lane & (G - 1), g = lane / G, gbase = lane & ~(G - 1);
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t *sc = scratch[threadIdx.x >> 5];

  uint32_t wq[kOwn];  // the exponents of this lane's slots
#pragma unroll
  for (int k = 0; k < kOwn; ++k) wq[k] = fx_weights(own_slot(k, lg));

  // this warp's cells: an equal share of the work, counted as particles plus
  // kGCellWork a cell (work of the cells before c: off[c] + kGCellWork c)
  const int64_t base0 = off[0], total = off[n_cells] - base0 + kGCellWork * n_cells;
  auto share = [&](int64_t k) { return base0 + (total / nwarps) * k + (total % nwarps) * k / nwarps; };
  const int64_t Lx = lower_bound16_by([&](int64_t c) { return off[c] + kGCellWork * c; }, n_cells,
                                      share(lane < 16 ? warp : warp + 1), lane);
  // (whole tasks: a share of nine cells would be three tasks of four, four and one)
  const int64_t whole = min((Lx + kCells - 1) / kCells * kCells, n_cells);
  const int64_t ca = __shfl_sync(0xffffffffu, whole, 0), cb = __shfl_sync(0xffffffffu, whole, 16);
  for (int64_t c0 = ca; c0 < cb; c0 += 32) {
    const int ncell = (int)(cb - c0 < 32 ? cb - c0 : 32);
    // rank the run's cells by size, largest first (bitonic; lane l's cell is
    // c0 + l, absent cells last)
    const int64_t o_l = off[c0 + (lane < ncell ? lane : ncell)];
    const int64_t o_n = lane < ncell ? off[c0 + lane + 1] : o_l;
    const int64_t n_l = o_n - o_l;
    uint32_t key = lane < ncell ? ((uint32_t)(n_l < (1 << 26) ? n_l + 1 : 1 << 26) << 5) | (uint32_t)lane : (uint32_t)lane;
    if (ncell > kCells) {
#pragma unroll
      for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j >= 1; j >>= 1) {
          const uint32_t p = __shfl_xor_sync(0xffffffffu, key, j);
          const bool lower = (lane & j) == 0, up = (lane & k) == 0;
          key = (lower == up) ? max(key, p) : min(key, p);
        }
    }
    const double inv_l = n_l > 0 ? recip_count((int)n_l) : 0.0;  // of lane l's cell
    for (int r0 = 0; r0 < ncell; r0 += kCells) {
      const int src = (int)(__shfl_sync(0xffffffffu, key, (r0 + g) & 31) & 31u);
      const bool valid = r0 + g < ncell;
      const int64_t a = __shfl_sync(0xffffffffu, o_l, src), e = __shfl_sync(0xffffffffu, o_n, src);
      const int64_t c = c0 + src;
      const int n = valid ? (int)(e - a) : 0;
      const VT *px = v + a, *py = px + np, *pz = py + np;
      const int itmax = __reduce_max_sync(0xffffffffu, (n + G - 1) / G);

      // ---- pass A: the mean, and the range of the high words ----
      double sx = 0.0, sy = 0.0, sz = 0.0;
      int32_t lo0 = 0x7fffffff, lo1 = lo0, lo2 = lo0, hi0 = (int32_t)0x80000000, hi1 = hi0, hi2 = hi0;
      {
        const VT *qx = px + lg, *qy = py + lg, *qz = pz + lg;
        int left = n - lg;  // this lane's particles at left > 0, left > 8, ..
        for (int it = 0; it < itmax; it += kGAhead) {
          VT x[kGAhead], y[kGAhead], z[kGAhead];
#pragma unroll
          for (int k = 0; k < kGAhead; ++k)  // all loads first
            if (k * G < left) x[k] = __ldg(qx + k * G), y[k] = __ldg(qy + k * G), z[k] = __ldg(qz + k * G);
#pragma unroll
          for (int k = 0; k < kGAhead; ++k)
            if (k * G < left) {
              sx += (double)x[k];
              sy += (double)y[k];
              sz += (double)z[k];
              const int32_t k0 = fx_key(v_words(x[k]).x), k1 = fx_key(v_words(y[k]).x), k2 = fx_key(v_words(z[k]).x);
              lo0 = min(lo0, k0), hi0 = max(hi0, k0);
              lo1 = min(lo1, k1), hi1 = max(hi1, k1);
              lo2 = min(lo2, k2), hi2 = max(hi2, k2);
            }
          qx += kGAhead * G, qy += kGAhead * G, qz += kGAhead * G;
          left -= kGAhead * G;
        }
      }
      const double inv_n = __shfl_sync(0xffffffffu, inv_l, src);
      // lane lg of the group holds component lg & 3
      const double U = group_scatter3<G>(sx, sy, sz, 0.0, lg, [](double p, double q) { return p + q; }) * inv_n;
      const int32_t klo = group_scatter3<G>(lo0, lo1, lo2, 0, lg, [](int32_t p, int32_t q) { return min(p, q); });
      const int32_t khi = group_scatter3<G>(hi0, hi1, hi2, 0, lg, [](int32_t p, int32_t q) { return max(p, q); });
      uint32_t mh;
      const bool ranged = fx_range(U, klo, khi, mh) && (sizeof(VT) == 8 || fx_exp(mh) >= kFxMinExpF);
      const bool fixed = (ranged && n > kGFew) || (lg & 3) == 3;
      const uint2 uw = v_words(U);
      const uint64_t Uf = fx_from_words(uw.x, uw.y, fx_exp(mh) + kFxHead + 1023);
      const unsigned okmask = __ballot_sync(0xffffffffu, fixed);
      bool fx = ((~okmask >> gbase) & (0xffffffffu >> (32 - G))) == 0u;  // the whole cell
      const int fold = fx_fold_bits((n + G - 1) / G);
      const FxCell cell = fx_cell(__shfl_sync(0xffffffffu, mh, gbase), __shfl_sync(0xffffffffu, mh, gbase + 1),
                                  __shfl_sync(0xffffffffu, mh, gbase + 2));

      double val[kOwn] = {};  // the sums of this lane's slots
      // ---- pass B ----
      {
        const uint64_t U0 = __shfl_sync(0xffffffffu, (unsigned long long)Uf, gbase),
                       U1 = __shfl_sync(0xffffffffu, (unsigned long long)Uf, gbase + 1),
                       U2 = __shfl_sync(0xffffffffu, (unsigned long long)Uf, gbase + 2);
        const int t0 = cell.e[0] + kFxHead + 1023, t1 = cell.e[1] + kFxHead + 1023, t2 = cell.e[2] + kFxHead + 1023;
        const int nf = fx ? n : 0;
        const int itfx = __reduce_max_sync(0xffffffffu, (nf + G - 1) / G);
        for (int b0 = 0; b0 < itfx; b0 += kFxBlock) {
          FxSums<kM6> S;
          const int b1 = min(b0 + kFxBlock, itfx);
          // (loads one particle ahead)
          const VT *qx = px + b0 * G + lg, *qy = py + b0 * G + lg, *qz = pz + b0 * G + lg;
          int left = nf - b0 * G - lg;
          S.clear(max(0, min(kFxBlock, (left + G - 1) / G)), fold);
          VT x = VT(0), y = VT(0), z = VT(0);
          if (left > 0) x = __ldg(qx), y = __ldg(qy), z = __ldg(qz);
#pragma unroll 1
          for (int it = b0; it < b1; ++it) {
            if (it == b0 + kFxMid) S.carry();
            const uint2 wx = v_words(x), wy = v_words(y), wz = v_words(z);
            qx += G, qy += G, qz += G;
            if (left > G) x = __ldg(qx), y = __ldg(qy), z = __ldg(qz);
            const bool in = left > 0;  // a lane past its cell adds c = 0
            left -= G;
            fx_accumulate<kM6>(S, in ? fx_offset(fx_from_words(wx.x, wx.y, t0), U0) : 0,
                               in ? fx_offset(fx_from_words(wy.x, wy.y, t1), U1) : 0,
                               in ? fx_offset(fx_from_words(wz.x, wz.y, t2), U2) : 0, cell);
          }
          double f[kOwn];
          group_transpose<G, int64_t>([&](int q) { return fx_fold<kM6>(S, q, fold); }, f, sc, lane);
#pragma unroll
          for (int k = 0; k < kOwn; ++k) val[k] = b0 == 0 ? f[k] : val[k] + f[k];
        }
      }
      {  // heavy tails: lane i < 3 of the group owns u_ii (slots 0, 3, 5) and w_ii
        const uint32_t hu = (uint32_t)__double2hiint(lg == 0 ? val[0] : val[1]);
        const uint32_t hw = (uint32_t)__double2hiint(lg == 0 ? val[2] : val[3]);
        const int32_t lu = fx_log(hu, lg == 0 ? cell.e[0] : lg == 1 ? cell.e[1] : cell.e[2], fold);
        const int32_t lmax = max(__shfl_sync(0xffffffffu, lu, gbase),
                                 max(__shfl_sync(0xffffffffu, lu, gbase + 1), __shfl_sync(0xffffffffu, lu, gbase + 2)));
        const uint32_t hn = (2u * 1023u << 20) - (uint32_t)__double2hiint(inv_n);  // of n
        const unsigned heavy = __ballot_sync(0xffffffffu, lg < 3 && fx_heavy(hw, hu, hn, cell.er, lmax));
        fx = fx && ((heavy >> gbase) & 7u) == 0u;
      }
      if (!__all_sync(0xffffffffu, fx || n == 0)) {  // some cell of the task in FP64
        const double Ux = __shfl_sync(0xffffffffu, U, gbase), Uy = __shfl_sync(0xffffffffu, U, gbase + 1),
                     Uz = __shfl_sync(0xffffffffu, U, gbase + 2);
        double t[kNSum];
#pragma unroll
        for (int q = 0; q < kNSum; ++q) t[q] = 0.0;
        const int itd = __reduce_max_sync(0xffffffffu, fx ? 0 : (n + G - 1) / G);
        for (int it = 0, i = lg; it < itd; ++it, i += G)
          if (!fx && i < n) accumulate26d(t, (double)__ldg(px + i) - Ux, (double)__ldg(py + i) - Uy, (double)__ldg(pz + i) - Uz);
        double d[kOwn];
        group_transpose<G, double>([&](int q) { return t[q]; }, d, reinterpret_cast<double *>(sc), lane);
#pragma unroll
        for (int k = 0; k < kOwn; ++k) val[k] = fx ? val[k] : d[k];
      }
      // ---- means, written by the slots' lanes ----
      double out[kOwn];
#pragma unroll
      for (int k = 0; k < kOwn; ++k) {
        // inv_n 2^s: a normal double times a power of two, exact
        const int s = fx ? fx_exponent(wq[k], cell, fold) : 0;
        out[k] = val[k] * __hiloint2double(__double2hiint(inv_n) + (n > 0 ? s * (1 << 20) : 0), __double2loint(inv_n));
      }
      const double u11 = __shfl_sync(0xffffffffu, out[0], gbase), u22 = __shfl_sync(0xffffffffu, out[1], gbase + 1),
                   u33 = __shfl_sync(0xffffffffu, out[1], gbase + 2);
      if (valid) {
        double *mo = mom + c * FP_NMOM;
        if (lg < 8) {
#pragma unroll
          for (int k = 0; k < kOwn; ++k) {
            const int q = own_slot(k, lg);
            if (q < kNMomSum) mo[kU2 + q] = out[k];
            if (kM6 && q == kM6Sum) m6[c] = out[k];
          }
        }
        if (lg < 3) mo[kU + lg] = U;
        if (lg == 3) {
          mo[kN] = u2d_exact((uint32_t)n);
          mo[kTheta] = (u11 + u22 + u33) * (1.0 / 3.0);
        }
      }
    }
  }
}

template <typename VT, int G>
static void launch_g(const VT *v, int64_t np, const int64_t *off, int64_t n_cells, double *mom, double *m6,
                     cudaStream_t st, int sm_count) {
  int64_t blocks = (n_cells + (32 / G) * kGWarps - 1) / ((32 / G) * kGWarps);  // a task a warp at least
  if (blocks > (int64_t)sm_count * kGBlocksPerSm) blocks = (int64_t)sm_count * kGBlocksPerSm;
  if (m6)
    gather_fp64_kernel<VT, true, G><<<(unsigned)blocks, 32 * kGWarps, 0, st>>>(v, np, off, n_cells, mom, m6);
  else
    gather_fp64_kernel<VT, false, G><<<(unsigned)blocks, 32 * kGWarps, 0, st>>>(v, np, off, n_cells, mom, m6);
}

template <typename VT>
static void launch_t(const VT *v, int64_t np, const int64_t *off, int64_t n_cells, int64_t whole, double *mom,
                     double *m6, cudaStream_t st, int sm_count) {
  // a whole warp a cell while every cell has a resident warp of its own (the
  // time is one cell's chain then: 400 cells of 100 particles 9.7 us, 14.5
  // with eight lanes); beyond, eight lanes (16: 461 us against 411 on 131,072
  // cells of 91 particles, 4: 510).  A part of a larger call takes the whole's
  // form: the two add in different orders, and a cell's bits do not depend on the
  // parts that its call is cut into.
  if (whole <= (int64_t)sm_count * kGBlocksPerSm * kGWarps)
    launch_g<VT, 32>(v, np, off, n_cells, mom, m6, st, sm_count);
  else
    launch_g<VT, 8>(v, np, off, n_cells, mom, m6, st, sm_count);
}

// whole: the cells of the call that these n_cells are a part of
void launch_gather_fp64(const void *v, int v_dtype, int64_t np, const int64_t *off, int64_t n_cells, int64_t whole,
                        double *mom, double *m6, cudaStream_t st, int sm_count) {
  if (v_dtype == FP_V_F32)
    launch_t<float>((const float *)v, np, off, n_cells, whole, mom, m6, st, sm_count);
  else
    launch_t<double>((const double *)v, np, off, n_cells, whole, mom, m6, st, sm_count);
}

}  // namespace fpc
