// adjoint.cu -- reverse mode through the exact closure (implicit function
// of Eq. system9x9) and through the moment gather, for sm_103a.
//
// With F(m, Y) = A(m) Y - r(m) = 0 defining the coefficients Y(m), a loss
// gradient gY = dL/dY pulls back to the moments as
//     lambda = A^-T gY,       dL/dm = -(dF/dm)^T lambda,
// and to the particle velocities through m_k = <psi_k(c)>, c = v - U:
//     dL/dv_p = (1/N) sum_k gm_k (grad psi_k(c_p) - <grad psi_k>) + gm_U / N.
//
// Kernel 1 (one thread per cell, FP64): lambda from the forward solve's
// stored factors (two triangular solves) or, without them, by re-assembling
// A and eliminating A^T with partial pivoting; then -lambda is propagated
// back through the assembly formulas by hand-written reverse mode.  Kernel 2
// (equal slices of the particles, 32 cells' tables at a time): the
// per-particle polynomial above, in the velocity's precision, one pass over
// the particles.
#include <climits>
#include <cstdint>

#include "closure_math.cuh"
#include "fp_device.cuh"
#include "quads.cuh"

namespace fpc {

// gm += -(dF/dm)^T lambda for F(m, Y) = A(m) Y - r(m) (the assembly of
// Eq. system9x9 differentiated by hand), with u, w, u3 adjoints kept per full
// index and folded onto the symmetric moment slots at the end.  Every factor
// that does not depend on the row's lambda is formed once per cell, so each
// term costs one FMA on the (scarce) FP64 pipe.
//   stress rows (ij): F = sum_k (C_ik u_kj + C_jk u_ki) + G_i b_j + G_j b_i
//                         + (2 / tau) u_ij - 2 e2 w_ij
//   heat rows (i):    F = sum_l C_il b_l + 2 sum_kl C_kl u_ikl + G_i (s4 - 9 th^2)
//                         + 2 sum_k G_k (w_ki - 3 th u_ki) + (4 / (3 tau)) b_i
//                         - e2 (3 z_i - 3 th b_i - 2 sum_k u_ik b_k)
// with b_i = sum_k u_ikk, s4 = sum_k w_kk, e2 = eps2_hat / (tau th).  With
// kAdd the results are added to gm, else they are stored in the 26 slots they
// fill (the N and U slots are left as they are).
template <bool kAdd>
__host__ __device__ __forceinline__ void assembly_vjp(const double (&m)[FP_NMOM], const double (&Y)[9],
                                                      const double (&lam)[9], double tc, double eps2_hat,
                                                      double (&gm)[FP_NMOM]) {
  double C[3][3], G[3], u[3][3], w[3][3], b[3], z[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    G[i] = Y[6 + i];
    z[i] = m[kZ + i];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      C[i][j] = Y[sym2(i, j)];
      u[i][j] = m[kU2 + sym2(i, j)];
      w[i][j] = m[kW + sym2(i, j)];
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) b[i] = m[kU3 + sym3(i, 0, 0)] + m[kU3 + sym3(i, 1, 1)] + m[kU3 + sym3(i, 2, 2)];
  const double th = m[kTheta];
  const double itau = rcp_d(tc), ith = rcp_d(th);
  const double e2 = eps2_hat * itau * ith;
  // per-cell factors of the row adjoints
  const double itau2 = times_pow2<1>(itau), e2x2 = times_pow2<1>(e2), me2x2 = -e2x2, mz = -3.0 * e2;
  const double kb = fma(4.0 / 3.0, itau, 3.0 * e2 * th);  // heat row i on b_i
  const double m18th = -18.0 * th, m6th = -6.0 * th, e2x3 = 3.0 * e2, th3 = 3.0 * th;
  double G2[3], G6[3], eb2[3], P[3], E[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    G2[k] = times_pow2<1>(G[k]);
    G6[k] = m6th * G[k];
    eb2[k] = e2x2 * b[k];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    // heat row i on theta: -18 th G_i - 6 sum_k G_k u_ki + 3 e2 b_i;
    // on e2: -(3 z_i - 3 th b_i - 2 sum_k u_ik b_k)
    const double gu = fma(G[0], u[0][i], fma(G[1], u[1][i], G[2] * u[2][i]));
    const double ubs = fma(u[i][0], b[0], fma(u[i][1], b[1], u[i][2] * b[2]));
    P[i] = fma(m18th, G[i], fma(-6.0, gu, e2x3 * b[i]));
    E[i] = fma(2.0, ubs, fma(th3, b[i], -3.0 * z[i]));
  }
  double ub[3][3] = {}, wb[3][3] = {}, u3b[10] = {}, zb[3], bb[3] = {};
  double thb = 0.0, s4b = 0.0, e2b = 0.0, sw = 0.0;
  // stress rows
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const double f = -lam[sym2(i, j)];
      if (i == j) {  // the two terms of each sum are the same
        const double f2 = times_pow2<1>(f);
#pragma unroll
        for (int k = 0; k < 3; ++k) ub[k][i] = fma(f2, C[i][k], ub[k][i]);
        bb[i] = fma(f2, G[i], bb[i]);
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          ub[k][j] = fma(f, C[i][k], ub[k][j]);
          ub[k][i] = fma(f, C[j][k], ub[k][i]);
        }
        bb[j] = fma(f, G[i], bb[j]);
        bb[i] = fma(f, G[j], bb[i]);
      }
      ub[i][j] = fma(f, itau2, ub[i][j]);
      wb[i][j] = fma(f, me2x2, wb[i][j]);
      sw = fma(f, w[i][j], sw);  // e2 adjoint: -2 sum f w_ij
    }
  // heat-flux rows
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double f = -lam[6 + i], f2 = times_pow2<1>(f), f4 = times_pow2<2>(f), fe = e2x2 * f;
#pragma unroll
    for (int l = 0; l < 3; ++l) bb[l] = fma(f, C[i][l], bb[l]);
    // 2 sum_kl C_kl u_ikl: a slot with k != l collects (k, l) and (l, k)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      u3b[sym3(i, k, k)] = fma(f2, C[k][k], u3b[sym3(i, k, k)]);
#pragma unroll
      for (int l = k + 1; l < 3; ++l) u3b[sym3(i, k, l)] = fma(f4, C[k][l], u3b[sym3(i, k, l)]);
    }
    s4b = fma(f, G[i], s4b);
    thb = fma(f, P[i], thb);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wb[k][i] = fma(f, G2[k], wb[k][i]);
      ub[k][i] = fma(f, G6[k], ub[k][i]);
      ub[i][k] = fma(f, eb2[k], ub[i][k]);
      bb[k] = fma(fe, u[i][k], bb[k]);
    }
    bb[i] = fma(f, kb, bb[i]);
    zb[i] = f * mz;
    e2b = fma(f, E[i], e2b);
  }
  // e2 = eps2_hat / (tau th);  b_i = sum_k u_ikk;  s4 = sum_k w_kk
  e2b = fma(-2.0, sw, e2b);
  thb = fma(e2b, -e2 * ith, thb);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) u3b[sym3(i, k, k)] += bb[i];
#pragma unroll
  for (int k = 0; k < 3; ++k) wb[k][k] += s4b;
  // fold onto the moment slots
  auto put = [&](int k, double v) {
    if (kAdd)
      gm[k] += v;
    else
      gm[k] = v;
  };
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      put(kU2 + sym2(i, j), i != j ? ub[i][j] + ub[j][i] : ub[i][j]);
      put(kW + sym2(i, j), i != j ? wb[i][j] + wb[j][i] : wb[i][j]);
    }
#pragma unroll
  for (int q = 0; q < 10; ++q) put(kU3 + q, u3b[q]);
#pragma unroll
  for (int i = 0; i < 3; ++i) put(kZ + i, zb[i]);
  put(kTheta, thb);
}

template <bool kLU>
__device__ __forceinline__ void adjoint_cell(int64_t c, const double *__restrict__ mom,
                                             const double *__restrict__ coeffs, const int32_t *__restrict__ flags,
                                             const double *__restrict__ lu, const double *__restrict__ tau,
                                             const double *__restrict__ gY, const double *__restrict__ gm_in,
                                             double eps2_hat, double *__restrict__ gm_out) {
  double gm[FP_NMOM];
#pragma unroll
  for (int k = 0; k < FP_NMOM; ++k) gm[k] = gm_in ? gm_in[c * FP_NMOM + k] : 0.0;
  const int fl = flags[c];
  if (!(fl & (FP_FLAG_FEW | FP_FLAG_SINGULAR | FP_FLAG_NONFINITE))) {
    double m[FP_NMOM];
#pragma unroll
    for (int k = 0; k < FP_NMOM; ++k) m[k] = mom[c * FP_NMOM + k];
    const double tc = tau[c];
    // lambda = A^-T gY: with the forward's factors two triangular solves,
    // else eliminate the transposed augmented system
    double lam[9];
    if (kLU) {
      double g[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) g[i] = gY[c * 9 + i];
      lu_solve_transposed(lu + lu_base(c), g, lam);
    } else {
      double a[9][10];
      assemble(m, tc, eps2_hat, a);
      double at[9][10];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
#pragma unroll
        for (int j = 0; j < 9; ++j) at[i][j] = a[j][i];
        at[i][9] = gY[c * 9 + i];
      }
      double rinv[9];
      uint64_t perm;
      pivoted_solve<false, true>(at, 0.0, lam, rinv, perm);
    }
    double Y[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) Y[q] = coeffs[c * 9 + q];
    if (gm_in)
      assembly_vjp<true>(m, Y, lam, tc, eps2_hat, gm);
    else
      assembly_vjp<false>(m, Y, lam, tc, eps2_hat, gm);
  }
#pragma unroll
  for (int k = 0; k < FP_NMOM; ++k) gm_out[c * FP_NMOM + k] = gm[k];
}

// One thread per cell, grid-stride, FP64-bound (see solve_kernel; 306
// instructions a cell with the factors, 72 us of 131,072 cells).  With the
// factors three 128-thread blocks per SM, for the loads of the factors: 82 us,
// 89 with two capped at 128 registers and the FP64 reciprocals, 90 with four
// today.  Without them two blocks and no cap: 16,384 cells 29.8 us, 33 with
// the cap.
template <bool kLU>
__global__ void __launch_bounds__(128, kLU ? 3 : 2) adjoint_cell_kernel(const double *__restrict__ mom,
                                                              const double *__restrict__ coeffs,
                                                              const int32_t *__restrict__ flags,
                                                              const double *__restrict__ lu,
                                                              const double *__restrict__ tau,
                                                              const double *__restrict__ gY,
                                                              const double *__restrict__ gm_in, int64_t n_cells,
                                                              double eps2_hat, double *__restrict__ gm_out) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cells;
       c += (int64_t)gridDim.x * blockDim.x)
    adjoint_cell<kLU>(c, mom, coeffs, flags, lu, tau, gY, gm_in, eps2_hat, gm_out);
}

// ---------------------------------------------------------------------------
// particle gradient
// ---------------------------------------------------------------------------
template <typename T>
constexpr int kAConst = sizeof(T) == 4 ? 44 : 40;  // table entries per cell
constexpr int64_t kACellWork = 50;  // a cell's share of building a chunk's table, in particles (24: 98 us, 100: 98, 50: 94)

// Per-cell table of the particle polynomial, every coefficient with its
// multiplicity.  With c = v - U, r2 = |c|^2 and
//   s_d = W_d . c + r2 z_d,    t = c . s + 3 r2 (z . c)
//   N dL/dv_d = B_d + sum_j c_j (Mu_dj + sum_{k >= j} A_{d,jk} c_k) + c_d t + r2 s_d
// (Mu from gm_u and gm_theta, A from gm_u3, W from gm_w, z from gm_z;
// B = gm_U minus the cell mean of the rest).  In nearly singular cells these terms
// cancel to a thousandth and less, so in FP32 what each of them loses shows:
//   - U is a pair (v - U rounded at |U| would be off by that over |c|);
//   - the division by N comes last, not into every coefficient;
//   - B, a sum of 27 products a component, is summed with its rounding errors.
// (Each cell's gradient against 64 bits, the worst cells of eight cylinder
// populations: 5.4e-7 in the geometric mean, 8.3e-7 with none of the three, 7.4e-7
// without the pair.)  In FP64 the coefficients are divided by N.
enum { AA3 = 0, AW = 18, AZ = 24, AMU = 28, AU = 34, AB = 37, AUL = 40, AIN = 43 };

// a sum of products, in FP32 with its rounding errors
template <typename T>
struct ProductSum {
  T h;
  __device__ __forceinline__ void mac(T a, T b) { h = tfma(a, b, h); }
  __device__ __forceinline__ T value() const { return h; }
};
template <>
struct ProductSum<float> {
  float h, l = 0.f;
  __device__ __forceinline__ void mac(float a, float b) {
    const float t = fmaf(a, b, h);
    l += fmaf(a, b, h - t);  // (exact where |a b| <= |h|; two-sum: 3 us more, the same errors)
    h = t;
  }
  __device__ __forceinline__ float value() const { return h + l; }
};

// One cell's table row by one lane, from its moment gradients (first half)
// and its moments (second half) staged in T.
template <typename T>
struct ParticleRow {
  T inv_n, Mu[6];
  ProductSum<T> B[3];

  // over N, in FP64
  __device__ __forceinline__ T part(T x) const { return sizeof(T) == 4 ? x : x * inv_n; }

  __device__ __forceinline__ void gradients(const T *gc, int n, T *row) {
    inv_n = n > 0 ? T(1) / T(n) : T(0);
    T r[28];
    // d/dc_d of the slot's monomial: 3 c^2 (111), 2 c_j c_k and c_j^2 (112), c_j c_k (123)
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = j; k < 3; ++k)
          r[AA3 + 6 * d + sym2(j, k)] = T(1 + (j == d) + (k == d)) * part(gc[kU3 + sym3(d, j, k)]);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const bool diag = s == 0 || s == 3 || s == 5;
      r[AW + s] = (diag ? T(2) : T(1)) * part(gc[kW + s]);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) r[AZ + d] = part(gc[kZ + d]);
    r[27] = T(0);
    store_row(row, r);
    const T gth = part(gc[kTheta]) * T(2.0 / 3.0);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      const bool diag = s == 0 || s == 3 || s == 5;
      Mu[s] = diag ? tfma(T(2), part(gc[kU2 + s]), gth) : part(gc[kU2 + s]);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) B[d].h = part(gc[kU + d]);
  }

  // B less the cell mean of the polynomial, from the moments; U: the means in FP64
  __device__ __forceinline__ void moments(const T *mc, const double *U, T *row) {
    T u3[10];
#pragma unroll
    for (int s = 0; s < 10; ++s) u3[s] = mc[kU3 + s];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = j; k < 3; ++k) {
        const T u = mc[kU2 + sym2(j, k)], w = mc[kW + sym2(j, k)];
        const T Wjk = row[AW + sym2(j, k)] * (j == k ? T(1) : T(2));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          B[d].mac(-row[AA3 + 6 * d + sym2(j, k)], u);
          B[d].mac(-Wjk, u3[sym3(d, j, k)]);
        }
        B[j].mac(T(-4) * row[AZ + k], w);
        if (j != k) B[k].mac(T(-4) * row[AZ + j], w);
      }
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          B[d].mac(-row[AZ + d], mc[kW + sym2(j, j)]);
#pragma unroll
          for (int k = 0; k < 3; ++k) B[d].mac(-row[AW + sym2(d, j)], u3[sym3(j, k, k)]);
        }
    } else {  // (fewer operations: the sums over k, and of the w_kk, first)
      const T s4 = mc[kW] + mc[kW + 3] + mc[kW + 5];
      T b[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) b[i] = u3[sym3(i, 0, 0)] + u3[sym3(i, 1, 1)] + u3[sym3(i, 2, 2)];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int j = 0; j < 3; ++j) B[d].mac(-row[AW + sym2(d, j)], b[j]);
        B[d].mac(-s4, row[AZ + d]);
      }
    }
    T u[3] = {mc[kU], mc[kU + 1], mc[kU + 2]};
    if constexpr (sizeof(T) == 4) {
      float r[4];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double x = U[d];
        r[d] = 0.f;
        if ((((uint32_t)__double2hiint(x) >> 20) & 0x7ffu) - (1023u - 100u) < 200u) {  // of f2_split
          const F2 s = f2_split(x);
          u[d] = s.h;
          r[d] = s.l;
        }
      }
      r[3] = inv_n;
      store_row(row + AUL, r);
    }
    const T r[12] = {Mu[0], Mu[1], Mu[2], Mu[3], Mu[4], Mu[5], u[0], u[1], u[2], B[0].value(), B[1].value(), B[2].value()};
    store_row(row + AMU, r);
  }
};

// Every warp of a resident grid takes an equal share of the work and walks its
// cells in chunks of up to 32: lane l builds the table row of the
// chunk's cell l, then the warp streams the chunk's particles in quads of
// four consecutive ones, with vector loads and stores where the arrays'
// alignment allows, the next quad loaded while one is computed, and one table
// row loaded a quad (another where a quad crosses a cell).  Bound: FP32 by the
// loads in flight and the tables' building (11.9M particles of 131,072 cells
// 114 us with eight lanes a cell and three 4-byte loads a particle, 90 now, 83
// without the terms that hold its error down; 288 MB at the copy rate: 42); FP64 by its pipe, 59 operations a particle (75
// before, and the table was built eight lanes a cell): 819,200 particles
// 212 -> 107 us (the operations alone: 96).  Registers: FP32 96 or 168 a
// thread 102 / 92 us, FP64 168 a thread 112.
template <typename VT>
__global__ void __launch_bounds__(sizeof(VT) == 4 ? 128 : 64, 4)
    adjoint_particle_kernel(const VT *__restrict__ v, int64_t np, const int64_t *__restrict__ off, int64_t n_cells,
                            const double *__restrict__ mom, const double *__restrict__ gm, VT *__restrict__ gv,
                            int vec) {
  using T = VT;
  constexpr int kW = sizeof(VT) == 4 ? 4 : 2;     // warps per block
  constexpr int kRow = sizeof(VT) == 4 ? 44 : 42;  // table row stride: 16-byte accesses of eight rows hit all banks
  constexpr int kIn = FP_NMOM | 1;
  __shared__ __align__(16) T table[kW][32 * kRow];
  __shared__ T stages[kW][32 * kIn];
  __shared__ int cofs[kW][33];  // the chunk's cell starts, relative to its first particle
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const uint32_t warp = blockIdx.x * kW + wib, nwarps = gridDim.x * kW;
  T *tab = table[wib], *stage = stages[wib];
  int *co = cofs[wib];
  const Share sh = warp_share(off, n_cells, kACellWork, warp, nwarps, lane);
  const int64_t tA = sh.p0, tB = sh.p1, cb = sh.c1;

  for (int64_t cbase = sh.first; cbase < cb; cbase += 32) {
    const int64_t c = cbase + lane;
    const bool valid = c < cb;
    const int64_t a0 = off[valid ? c : cb];
    const int64_t a1 = valid ? off[c + 1] : a0;
    // the chunk's particle range, clipped to the slice
    const int64_t o0 = max(__shfl_sync(0xffffffffu, a0, 0), tA);
    const int64_t oe = min(__shfl_sync(0xffffffffu, a1, 31), tB);
    const int i4 = (int)max(oe - o0, (int64_t)0);
    co[lane] = (int)min(max(a0 - o0, (int64_t)0), (int64_t)i4);
    if (lane == 31) co[32] = i4;
    // ---- the chunk's particles, in quads (quad Q: particles 4Q .. 4Q + 3) ----
    const int64_t Qs = o0 >> 2, Qe = i4 > 0 ? (o0 + i4 + 3) >> 2 : Qs;
    const VT *px = v + o0, *py = px + np, *pz = py + np;
    VT *qx = gv + o0, *qy = qx + np, *qz = qy + np;
    // (a lane's first quad is loaded before the table is built, the next ones
    // each while one is computed)
    T nx[4], ny[4], nz[4];
    auto load = [&](int qb) {
      if (qb >= 0 && qb + 4 <= i4) {
        load_comp(px + qb, vec & 3, nx);
        load_comp(py + qb, (vec >> 2) & 3, ny);
        load_comp(pz + qb, (vec >> 4) & 3, nz);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int q = qb + u;
          nx[u] = ny[u] = nz[u] = T(0);
          if ((unsigned)q < (unsigned)i4) {
            nx[u] = px[q];
            ny[u] = py[q];
            nz[u] = pz[q];
          }
        }
      }
    };
    const int qe = (int)((Qe << 2) - o0);
    int qb = (int)(((Qs + lane) << 2) - o0);  // chunk index of the quad's first particle
    if (qb < qe) load(qb);
    {
      const int ncell = (int)min(cb - cbase, (int64_t)32);
      ParticleRow<T> r;
      const bool both = ncell <= 16;  // both sets of rows fit the stage at once
      stage_rows<FP_NMOM>(gm + cbase * FP_NMOM, ncell, stage, lane, both ? mom + cbase * FP_NMOM : nullptr, 16 * kIn);
      __syncwarp();
      if (valid) r.gradients(stage + lane * kIn, (int)(a1 - a0), tab + lane * kRow);
      if (!both) {
        __syncwarp();
        stage_rows<FP_NMOM>(mom + cbase * FP_NMOM, ncell, stage, lane);
        __syncwarp();
      }
      if (valid) r.moments(stage + (lane + (both ? 16 : 0)) * kIn, mom + c * FP_NMOM + kU, tab + lane * kRow);
    }
    __syncwarp();
    for (; qb < qe; qb += 128) {
      const bool whole = qb >= 0 && qb + 4 <= i4;
      T mx[4], my[4], mz[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        mx[u] = nx[u];
        my[u] = ny[u];
        mz[u] = nz[u];
      }
      if (qb + 128 < qe) load(qb + 128);
      // cell of the quad's first particle: the last cl with co[cl] <= max(qb, 0)
      const int q0 = max(qb, 0);
      int cl = 0;
#pragma unroll
      for (int st = 16; st >= 1; st >>= 1)
        if (co[cl + st] <= q0) cl += st;
      T K[kAConst<T>];
      load_row(tab + cl * kRow, K);
      int next = cl < 31 ? co[cl + 1] : INT_MAX;  // where the next cell starts
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // (particles outside the chunk are computed on zeros and not stored)
        const int q = qb + u;
        if (q >= next) {  // past a cell boundary (and any empty cells)
          while (cl < 31 && co[cl + 1] <= q) ++cl;
          load_row(tab + cl * kRow, K);
          next = cl < 31 ? co[cl + 1] : INT_MAX;
        }
        T cc[3] = {mx[u] - K[AU], my[u] - K[AU + 1], mz[u] - K[AU + 2]};
        if constexpr (sizeof(T) == 4) {
#pragma unroll
          for (int d = 0; d < 3; ++d) cc[d] -= K[AUL + d];
        }
        const T r2 = tfma(cc[0], cc[0], tfma(cc[1], cc[1], cc[2] * cc[2]));
        T s[3], out[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          s[d] = r2 * K[AZ + d];
#pragma unroll
          for (int j = 0; j < 3; ++j) s[d] = tfma(K[AW + sym2(d, j)], cc[j], s[d]);
        }
        const T zc = tfma(K[AZ], cc[0], tfma(K[AZ + 1], cc[1], K[AZ + 2] * cc[2]));
        const T t = tfma(T(3) * r2, zc, tfma(cc[0], s[0], tfma(cc[1], s[1], cc[2] * s[2])));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          T g = K[AB + d];
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            T h = K[AMU + sym2(d, j)];
#pragma unroll
            for (int k = j; k < 3; ++k) h = tfma(K[AA3 + 6 * d + sym2(j, k)], cc[k], h);
            g = tfma(cc[j], h, g);
          }
          out[d] = tfma(r2, s[d], tfma(cc[d], t, g));
          if constexpr (sizeof(T) == 4) out[d] *= K[AIN];
        }
        mx[u] = out[0];
        my[u] = out[1];
        mz[u] = out[2];
      }
      if (whole) {
        store_comp(qx + qb, vec & 3, mx);
        store_comp(qy + qb, (vec >> 2) & 3, my);
        store_comp(qz + qb, (vec >> 4) & 3, mz);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int q = qb + u;
          if ((unsigned)q < (unsigned)i4) {
            qx[q] = mx[u];
            qy[q] = my[u];
            qz[q] = mz[u];
          }
        }
      }
    }
    __syncwarp();  // the table and offsets are rewritten by the next chunk
  }
}

// ---- small problems ----
constexpr int kAG = 8;              // lanes per cell while building constants
constexpr int kACells = 32 / kAG;   // consecutive cells per warp task
constexpr int kAWarps = 8;          // warps per block
constexpr int kAGConst = 44;        // table entries per cell

// Per-cell table of the particle polynomial, every coefficient already
// multiplied by 1/N and by its constant factor:
//   dL/dv_d = Mu'_d.c + sum_{j<=k} A3'_{d,jk} c_j c_k
//             + c_d (c.W'c + |c|^2 gz'.c) + |c|^2 (W'c)_d + |c|^4 gz''_d + B_d
// with Mu' = Mu/N, A3'_{d,jk} = 3 m_jk A_{djk}/N (m = 1 on, 2 off the
// diagonal), W' = 2W/N, gz' = 4gz/N, gz'' = gz/N, B = (gm_U - <grad psi>)/N.
enum { GU = 0, GMU = 3, GA3 = 9, GW = 27, GGZ4 = 33, GGZ1 = 36, GB = 39 };

template <typename T>
__device__ __forceinline__ T shfl_g(T x, int src, int lane) {
  return __shfl_sync(0xffffffffu, x, (lane & ~(kAG - 1)) + src);
}

// multiplicity of a symmetric third-order slot (111: 1, 112: 3, 123: 6)
__host__ __device__ constexpr int mult3(int s) { return (s == 0 || s == 6 || s == 9) ? 1 : (s == 4 ? 6 : 3); }

// FP32 particles of small problems: a warp takes four consecutive cells; an
// 8-lane group folds its cell's moments and moment gradients into the 35
// coefficients of the per-particle polynomial (shared-memory table), then all
// 32 lanes walk the four cells' contiguous particle range.
__global__ void __launch_bounds__(32 * kAWarps, 3)
    adjoint_particle_group_kernel(const float *__restrict__ v, int64_t np, const int64_t *__restrict__ off,
                                  int64_t n_cells, const double *__restrict__ mom, const double *__restrict__ gm,
                                  float *__restrict__ gv) {
  using VT = float;
  using T = float;
  constexpr int G = kAG;
  __shared__ __align__(16) T table[kAWarps][kACells][kAGConst];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int lg = lane & (G - 1);
  const int g = lane / G;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const VT *vx = v, *vy = v + np, *vz = v + 2 * np;
  VT *gx = gv, *gy = gv + np, *gz = gv + 2 * np;
  T(*tab)[kAGConst] = table[wib];

  for (int64_t base = warp * kACells; base < n_cells; base += nwarps * kACells) {
    const int64_t c = base + g;
    const bool valid = c < n_cells;
    const int64_t a0 = off[valid ? c : n_cells];
    const int64_t e = valid ? off[c + 1] : a0;
    const int n = (int)(e - a0);
    // the cell's 30 moments and 30 moment gradients, converted once: lane lg
    // holds slots lg + 8 j of the concatenation [mom | gm] (60 values)
    T cv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int slot = lg + 8 * j;
      double x = 0.0;
      if (valid && slot < 60) x = slot < 30 ? mom[c * FP_NMOM + slot] : gm[c * FP_NMOM + slot - 30];
      cv[j] = (T)x;
    }
    {
      auto M_ = [&](int k) -> T { return shfl_g(cv[k / 8], k % 8, lane); };
      auto GM = [&](int k) -> T { return shfl_g(cv[(30 + k) / 8], (30 + k) % 8, lane); };
      // u-part: G_d += sum_j Mu_dj c_j with Mu_dj = gm_u(dj) (1 + delta_dj); theta adds 2/3 gm_theta c_d
      const T gth = GM(kTheta) * T(2.0 / 3.0);
      T Mu[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        const bool diag = s == 0 || s == 3 || s == 5;
        Mu[s] = GM(kU2 + s) * (diag ? T(2) : T(1)) + (diag ? gth : T(0));
      }
      // u3-part: G_d += 3 sum_jk A_djk c_j c_k with A = gm_u3(slot) / multiplicity
      T A3[10];
#pragma unroll
      for (int s = 0; s < 10; ++s) A3[s] = GM(kU3 + s) / T(mult3(s));
      // w-part: G_d += 2 c_d (c.W c) + 2 |c|^2 (W c)_d with W = gm_w(slot) / multiplicity
      T W[3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) W[i][j] = GM(kW + sym2(i, j)) * (i == j ? T(1) : T(0.5));
      // z-part: G_d += 4 |c|^2 c_d (gz.c) + |c|^4 gz_d
      const T gzv[3] = {GM(kZ), GM(kZ + 1), GM(kZ + 2)};
      // the cell mean of grad psi, from the moments
      T G0[3];
      {
        T u[3][3], w[3][3], b[3], u3[10];
#pragma unroll
        for (int s = 0; s < 10; ++s) u3[s] = M_(kU3 + s);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            u[i][j] = M_(kU2 + sym2(i, j));
            w[i][j] = M_(kW + sym2(i, j));
          }
#pragma unroll
        for (int i = 0; i < 3; ++i) b[i] = u3[sym3(i, 0, 0)] + u3[sym3(i, 1, 1)] + u3[sym3(i, 2, 2)];
        const T s4 = w[0][0] + w[1][1] + w[2][2];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          T acc = 0;
#pragma unroll
          for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k)
              acc += T(3) * A3[sym3(d, j, k)] * u[j][k] + T(2) * W[j][k] * u3[sym3(d, j, k)];
#pragma unroll
          for (int j = 0; j < 3; ++j) acc += T(2) * W[d][j] * b[j] + T(4) * gzv[j] * w[d][j];
          acc += s4 * gzv[d];
          G0[d] = acc;
        }
      }
      const T inv_n = n > 0 ? T(1) / T(n) : T(0);
      const T U0 = M_(kU), U1 = M_(kU + 1), U2 = M_(kU + 2);
      const T gU0 = GM(kU) * inv_n, gU1 = GM(kU + 1) * inv_n, gU2 = GM(kU + 2) * inv_n;
      if (lg == 0) {
        T *r = tab[g];
        r[GU] = U0;
        r[GU + 1] = U1;
        r[GU + 2] = U2;
#pragma unroll
        for (int s = 0; s < 6; ++s) r[GMU + s] = Mu[s] * inv_n;
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = j; k < 3; ++k)
              r[GA3 + 6 * d + sym2(j, k)] = A3[sym3(d, j, k)] * (j == k ? T(3) : T(6)) * inv_n;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = i; j < 3; ++j) r[GW + sym2(i, j)] = T(2) * W[i][j] * inv_n;
        const T gUv[3] = {gU0, gU1, gU2};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          r[GGZ4 + d] = T(4) * gzv[d] * inv_n;
          r[GGZ1 + d] = gzv[d] * inv_n;
          r[GB + d] = gUv[d] - G0[d] * inv_n;
        }
        r[GB + 3] = T(0);
        r[GB + 4] = T(0);
      }
    }
    const int64_t o0 = __shfl_sync(0xffffffffu, a0, 0);
    const int i1 = (int)(__shfl_sync(0xffffffffu, a0, 8) - o0);
    const int i2 = (int)(__shfl_sync(0xffffffffu, a0, 16) - o0);
    const int i3 = (int)(__shfl_sync(0xffffffffu, a0, 24) - o0);
    const int i4 = (int)(__shfl_sync(0xffffffffu, e, 24) - o0);
    const VT *px = vx + o0, *py = vy + o0, *pz = vz + o0;
    VT *qx = gx + o0, *qy = gy + o0, *qz = gz + o0;
    __syncwarp();
#pragma unroll 2
    for (int q = lane; q < i4; q += 32) {
      const int cl = (q >= i1) + (q >= i2) + (q >= i3);
      T K[kAGConst];
      load_row(tab[cl], K);
      const T cc[3] = {px[q] - K[GU], py[q] - K[GU + 1], pz[q] - K[GU + 2]};
      // the six products c_j c_k (j <= k), in sym2 order
      const T pr[6] = {cc[0] * cc[0], cc[0] * cc[1], cc[0] * cc[2], cc[1] * cc[1], cc[1] * cc[2], cc[2] * cc[2]};
      const T r2 = pr[0] + pr[3] + pr[5];
      const T r4 = r2 * r2;
      T Wc[3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
        Wc[i] = K[GW + sym2(i, 0)] * cc[0] + K[GW + sym2(i, 1)] * cc[1] + K[GW + sym2(i, 2)] * cc[2];
      const T t = cc[0] * Wc[0] + cc[1] * Wc[1] + cc[2] * Wc[2] +
                  r2 * (K[GGZ4] * cc[0] + K[GGZ4 + 1] * cc[1] + K[GGZ4 + 2] * cc[2]);
      T out[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        T gd = K[GMU + sym2(d, 0)] * cc[0] + K[GMU + sym2(d, 1)] * cc[1] + K[GMU + sym2(d, 2)] * cc[2];
#pragma unroll
        for (int s = 0; s < 6; ++s) gd += K[GA3 + 6 * d + s] * pr[s];
        out[d] = gd + cc[d] * t + r2 * Wc[d] + r4 * K[GGZ1 + d] + K[GB + d];
      }
      qx[q] = out[0];
      qy[q] = out[1];
      qz[q] = out[2];
    }
    __syncwarp();
  }
}

static int adj_sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 152;
  }
  return n;
}

// FP32 calls on up to this many cells take the group kernel: a table of four
// cells by eight lanes each is ready sooner than one of 32 by a lane each, and
// its small footprint runs beside other streams' kernels (16,384 cells of 50
// particles 11.9 us against 12.4; as a chunk of the host-resident step 26.6
// against 31; 40,000 cells of 50: 25.0 against 24.1).  The line is drawn by cells
// alone: with more particles a cell the other kernel is ahead below it already
// (16,384 cells of 150: 25.3 here, 19.8 there).
constexpr int64_t kGroupCells = 32768;

// A persistent grid (fewer blocks for small problems: two cells a warp at
// least).
template <typename VT>
static void launch_adjoint_particles(const VT *v, int64_t np, const int64_t *off, int64_t n_cells, const double *mom,
                                     const double *gm, VT *gv, cudaStream_t st) {
  if (sizeof(VT) == 4 && n_cells <= kGroupCells) {
    const int64_t cells_per_block = kAWarps * kACells, cap = (int64_t)adj_sm_count() * 8;
    int64_t blocks = (n_cells + cells_per_block - 1) / cells_per_block;
    if (blocks > cap) blocks = cap;
    adjoint_particle_group_kernel<<<(unsigned)blocks, 32 * kAWarps, 0, st>>>((const float *)v, np, off, n_cells, mom,
                                                                              gm, (float *)gv);
    return;
  }
  constexpr int kW = sizeof(VT) == 4 ? 4 : 2;
  static int per_sm = 0;
  if (!per_sm) {
    int k = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, adjoint_particle_kernel<VT>, 32 * kW, 0) != cudaSuccess ||
        k < 1)
      k = 1;
    per_sm = k;
  }
  int64_t blocks = (int64_t)adj_sm_count() * per_sm;
  const int64_t by_cells = (n_cells + 2 * kW - 1) / (2 * kW);
  if (blocks > by_cells) blocks = by_cells;
  if (blocks < 1) blocks = 1;
  adjoint_particle_kernel<VT>
      <<<(unsigned)blocks, 32 * kW, 0, st>>>(v, np, off, n_cells, mom, gm, gv, quad_classes(v, gv, np, 0, sizeof(VT)));
}

void launch_adjoint(const void *v, int v_dtype, int64_t np, const int64_t *off, int64_t n_cells, const double *tau,
                    double eps2_hat, const double *mom, const double *coeffs, const int32_t *flags, const double *lu,
                    const double *gY, const double *gm_in, double *gm_out, void *gv, cudaStream_t st) {
  {
    const int threads = 128;
    const int per_sm = lu ? 3 : 2;
    int64_t blocks = (n_cells + threads - 1) / threads;
    if (blocks > per_sm * adj_sm_count()) blocks = per_sm * adj_sm_count();
    if (lu)
      adjoint_cell_kernel<true><<<(unsigned)blocks, threads, 0, st>>>(mom, coeffs, flags, lu, tau, gY, gm_in,
                                                                      n_cells, eps2_hat, gm_out);
    else
      adjoint_cell_kernel<false><<<(unsigned)blocks, threads, 0, st>>>(mom, coeffs, flags, nullptr, tau, gY, gm_in,
                                                                       n_cells, eps2_hat, gm_out);
  }
  if (!gv) return;
  if (v_dtype == FP_V_F32)
    launch_adjoint_particles<float>((const float *)v, np, off, n_cells, mom, gm_out, (float *)gv, st);
  else
    launch_adjoint_particles<double>((const double *)v, np, off, n_cells, mom, gm_out, (double *)gv, st);
}

}  // namespace fpc
