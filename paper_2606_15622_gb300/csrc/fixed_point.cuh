// fixed_point.cuh -- the fixed-point arithmetic of the FP64 moment gather.
//
// GB300 issues one FP64 warp instruction every 64 cycles per SM sub-partition
// (68 measured) but one 32 x 32 + 64-bit integer multiply-add every 4 to 6, so
// the 26 central sums of a cell (61 FP64 flops a particle) are formed in
// integers: a component of c = v - U is an integer in units of 2^(E - 58), E the
// exponent with |c| < 2^E over the cell, held as two limbs h 2^29 + l,
// 0 <= l < 2^29.  A product that is only summed takes three multiply-adds into
// two 64-bit sums (h h', h l' + l h'); the dropped l l' is below 2^-58 of the
// largest product (<|c|^6> keeps it, the others its mean).  A product that is a
// factor again (c_i c_j, |c|^2, |c|^4) is rounded to 2^-58 of its largest value.
// Every component has its own exponent, and so has |c|^2 (the least power of
// two above the sum of the components' squared bounds), so a thin
// distribution keeps its digits.
//
// So a term is not exact but off by up to some 8 units of 2^-58 of the largest
// term that the bounds allow, where an FP64 term is rounded at 2^-53 of itself:
// closer than FP64 sums for Maxwellians, uniform cubes, beams and shock mixtures,
// less close where few particles lie far outside the others, which fx_heavy finds.
//
// Plain C++ but for the qualifiers: the host test compiles it with g++.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define FPC_HD __host__ __device__ __forceinline__
#else
#define FPC_HD inline
#endif

namespace fpc {

constexpr int kFxBits = 58;   // fraction bits: |c| < 2^58 units
constexpr int kFxLimb = 29;   // bits of the low limb
constexpr int kFxMid = 15;    // particles a lane sums before its middle sums (terms h l' + l h' < 2^59) are carried
constexpr int kFxBlock = 30;  // .. and before all its sums (terms < 2^58) are folded
constexpr int kFxFold = 3;    // bits a folded sum drops at most, so that ..
constexpr int kFxLanes = 8;   // .. the folded sums of so many lanes add up in 64 bits (more lanes: in FP64 from there)
static_assert(kFxBlock < 1 << (63 - kFxBits), "a lane's block of terms below 2^kFxBits");
static_assert(kFxLanes * kFxBlock < 1 << (63 - kFxBits + kFxFold), "the folded blocks of kFxLanes lanes");
// binades the largest |v| may lie above E (the mantissa, shifted to bit 63,
// is only ever shifted right)
constexpr int kFxHead = 63 - kFxBits;
constexpr int kFxMaxExp = 120;  // |E| accepted: 2^(5 E) and 2^(6 E) stay normal doubles
constexpr int kFxMinExpF = -67;  // of FP32 velocities: their subnormals, read as zero, are below half a unit

struct Fx {
  int32_t h, l;
};

// The bits to drop for a cell whose lanes sum up to m particles a block:
// kFxLanes m < 2^(63 - kFxBits + bits).  Dropping three always left the sums of
// cells of 30 particles by 32 lanes up to six times as far off as FP64 sums.
FPC_HD int fx_fold_bits(int m) {
  static_assert(kFxLanes == 8 && kFxFold == 3 && kFxBits == 58, "the steps below");
  return m < 4 ? 0 : m < 8 ? 1 : m < 16 ? 2 : kFxFold;
}

// a b + c, one instruction (written out: from the C++ the compiler makes
// 64 x 64-bit products of limbs that it has just widened)
FPC_HD int64_t fx_wide(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (int64_t)a * b + c;
#endif
}

FPC_HD Fx fx_split(int64_t c) {
  Fx r;
  r.h = (int32_t)(c >> kFxLimb);
  r.l = (int32_t)((uint32_t)c & ((1u << kFxLimb) - 1u));
  return r;
}

// a b in units of 2^-58, rounded (the mean of the dropped l l' put on)
constexpr int64_t kFxRound = ((int64_t)1 << (kFxLimb - 1)) + ((int64_t)1 << (kFxLimb - 2));
FPC_HD int64_t fx_mul(Fx a, Fx b) {
  const int64_t mid = fx_wide(a.h, b.l, fx_wide(a.l, b.h, kFxRound));
  return fx_wide(a.h, b.h, mid >> kFxLimb);
}
FPC_HD int64_t fx_sqr(Fx a) {
  const int64_t mid = fx_wide(a.h, 2 * a.l, kFxRound);
  return fx_wide(a.h, a.h, mid >> kFxLimb);
}

// Finite v = (-1)^s 1.f 2^e (the double's two words) in units of
// 2^(E - 58), modulo 2^64, truncated; top = E + kFxHead + 1023, e <= E + kFxHead.
// Zeros and subnormals (whose shift leaves nothing for an accepted E) give 0.
FPC_HD uint64_t fx_from_words(uint32_t hi, uint32_t lo, int top) {
  // the mantissa 1.f to bits 63 .. 11, then down by the binades to 2^(E + kFxHead)
  const uint64_t m = ((uint64_t)(hi | 0x00100000u) << 43) | ((uint64_t)lo << 11);
  const int r = top - (int)((hi >> 20) & 0x7ffu);
#ifdef __CUDA_ARCH__
  uint64_t u;
  asm("shr.u64 %0, %1, %2;" : "=l"(u) : "l"(m), "r"(r));  // amounts above 63 give 0
#else
  const uint64_t u = r > 63 ? 0 : m >> r;
#endif
  const uint64_t s = 0ull - (uint64_t)(hi >> 31);
  return (u ^ s) - s;
}
// c = v - U of such positions: they wrap, their difference is below 2^kFxBits
FPC_HD int64_t fx_offset(uint64_t v, uint64_t U) { return (int64_t)(v - U); }

// order of doubles on their high words: a signed key
FPC_HD int32_t fx_key(uint32_t hi) { return (int32_t)(hi ^ (uint32_t)(((int32_t)hi >> 31) & 0x7fffffff)); }
FPC_HD uint32_t fx_unkey(int32_t k) { return (uint32_t)(k ^ ((k >> 31) & 0x7fffffff)); }

FPC_HD uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
FPC_HD double fx_double(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t u = ((uint64_t)hi << 32) | lo;
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}

// A component whose values' high words lie between the keys klo and khi and
// whose mean is U: the high word of a bound on |v - U| (from the widened
// range, itself widened), and whether the fixed-point form takes it.  Refused:
// values that are not finite, all alike in their high words, more than
// 2^kFxHead times the spread from zero, or a spread beyond 2^+-kFxMaxExp.
FPC_HD int fx_exp(uint32_t mh) { return (int)(mh >> 20) - 1022; }  // E: the bound is < 2^E
FPC_HD bool fx_range(double U, int32_t klo, int32_t khi, uint32_t &mh) {
  const uint32_t wh = fx_unkey(khi), wl = fx_unkey(klo), uh = (uint32_t)(fx_bits(U) >> 32);
  const double vmax = fx_double(wh, wh >> 31 ? 0u : 0xffffffffu), vmin = fx_double(wl, wl >> 31 ? 0xffffffffu : 0u);
  const uint32_t a = (uint32_t)(fx_bits(vmax - U) >> 32) & 0x7fffffffu;
  const uint32_t b = (uint32_t)(fx_bits(U - vmin) >> 32) & 0x7fffffffu;
  mh = (a > b ? a : b) + 1;
  const int E = fx_exp(mh);
  // the largest exponent in sight (U rounds: it may lie a binade above every |v|)
  uint32_t vh = wh & 0x7fffffffu;
  if ((wl & 0x7fffffffu) > vh) vh = wl & 0x7fffffffu;
  if ((uh & 0x7fffffffu) > vh) vh = uh & 0x7fffffffu;
  return khi != klo && vh < 0x7ff00000u && (int)(vh >> 20) - 1023 <= E + kFxHead && E >= -kFxMaxExp && E <= kFxMaxExp;
}

// The exponents of a cell: E of each component, Er with |c|^2 < 2^Er from the
// bounds' high words (at least 2 E of each component, so that the alignment
// shifts are not negative), the shifts and what their floors lose on average.
struct FxCell {
  int e[3], er, sh[3], r2c;
};
FPC_HD FxCell fx_cell(uint32_t m0, uint32_t m1, uint32_t m2) {
  const uint32_t m[3] = {m0, m1, m2};
  FxCell c;
  int em = -100000;
  for (int d = 0; d < 3; ++d) {
    c.e[d] = fx_exp(m[d]);
    em = c.e[d] > em ? c.e[d] : em;
  }
  // sum of the squares of the bounds' leading 16 bits, rounded up, in units of 2^(2 em - 34)
  uint64_t s = 0;
  for (int d = 0; d < 3; ++d) {
    const int down = em - c.e[d];
    const uint32_t f = (((m[d] & 0xfffffu) | 0x100000u) >> 4) + 1;  // bound < f 2^(E - 17)
    const uint32_t g = (down > 16 ? 0u : f >> down) + 1;
    s += (uint64_t)g * g;
  }
#ifdef __CUDA_ARCH__
  const int top = 64 - __clzll((long long)s);
#else
  const int top = 64 - __builtin_clzll(s);
#endif
  c.er = 2 * em + (top > 34 ? top - 34 : 0);  // s < 2^top
  int k = 0;
  for (int d = 0; d < 3; ++d) {
    const int sh = c.er - 2 * c.e[d];
    c.sh[d] = sh > 62 ? 62 : sh;
    k += sh > 0;
  }
  c.r2c = (k + 1) >> 1;
  return c;
}

// The sums of one lane over up to kFxBlock particles, all in
// units of 2^-58.
// Slots: u_ij 0..5 (P), then 0..9 u_ijk, 10..15
// |c|^2 c_i c_j, 16..18 |c|^4 c_i, 19 |c|^6 as (hi, mid) pairs.
template <bool kM6>
struct FxSums {
  static constexpr int kN = kM6 ? 20 : 19;
  int64_t P[6], H[kN], M[kN], L;
  // for count particles to come: the mean of the dropped l l', 2^(2 kFxLimb - 2)
  // a term, goes into the middle sums beforehand (<|c|^6> sums its own), and
  // so do the halves that make the shifts of fx_fold round
  FPC_HD void clear(int count, int fold = kFxFold) {
    for (int q = 0; q < 6; ++q) P[q] = (1 << fold) >> 1;
    for (int q = 0; q < kN; ++q) {
      H[q] = (1 << fold) >> 1;
      M[q] = ((int64_t)(q == 19 ? 0 : count) << (kFxLimb - 2)) + ((int64_t)1 << (kFxLimb - 1));
    }
    L = 0;
  }
  // the middle sums' whole part into the high ones
  FPC_HD void carry() {
    for (int q = 0; q < kN; ++q) {
      H[q] += M[q] >> kFxLimb;
      M[q] &= ((int64_t)1 << kFxLimb) - 1;
    }
  }
};

FPC_HD void fx_mac(int64_t &H, int64_t &M, Fx a, Fx b) {
  H = fx_wide(a.h, b.h, H);
  M = fx_wide(a.l, b.h, fx_wide(a.h, b.l, M));
}

// One particle (c = 0: adds nothing that the rounding constants do not)
template <bool kM6>
FPC_HD void fx_accumulate(FxSums<kM6> &S, int64_t cx, int64_t cy, int64_t cz, const FxCell &cell) {
  const Fx x = fx_split(cx), y = fx_split(cy), z = fx_split(cz);
  const int64_t pxx = fx_sqr(x), pxy = fx_mul(x, y), pxz = fx_mul(x, z);
  const int64_t pyy = fx_sqr(y), pyz = fx_mul(y, z), pzz = fx_sqr(z);
  S.P[0] += pxx; S.P[1] += pxy; S.P[2] += pxz; S.P[3] += pyy; S.P[4] += pyz; S.P[5] += pzz;
  const Fx xx = fx_split(pxx), xy = fx_split(pxy), xz = fx_split(pxz);
  const Fx yy = fx_split(pyy), yz = fx_split(pyz), zz = fx_split(pzz);
  fx_mac(S.H[0], S.M[0], xx, x); fx_mac(S.H[1], S.M[1], xx, y); fx_mac(S.H[2], S.M[2], xx, z);
  fx_mac(S.H[3], S.M[3], yy, x); fx_mac(S.H[4], S.M[4], xy, z); fx_mac(S.H[5], S.M[5], zz, x);
  fx_mac(S.H[6], S.M[6], yy, y); fx_mac(S.H[7], S.M[7], yy, z); fx_mac(S.H[8], S.M[8], zz, y);
  fx_mac(S.H[9], S.M[9], zz, z);
  const Fx r2 = fx_split((pxx >> cell.sh[0]) + (pyy >> cell.sh[1]) + (pzz >> cell.sh[2]) + cell.r2c);
  fx_mac(S.H[10], S.M[10], r2, xx); fx_mac(S.H[11], S.M[11], r2, xy); fx_mac(S.H[12], S.M[12], r2, xz);
  fx_mac(S.H[13], S.M[13], r2, yy); fx_mac(S.H[14], S.M[14], r2, yz); fx_mac(S.H[15], S.M[15], r2, zz);
  const Fx r4 = fx_split(fx_sqr(r2));
  fx_mac(S.H[16], S.M[16], r4, x); fx_mac(S.H[17], S.M[17], r4, y); fx_mac(S.H[18], S.M[18], r4, z);
  if (kM6) {
    fx_mac(S.H[kM6 ? 19 : 0], S.M[kM6 ? 19 : 0], r4, r2);
    S.L = fx_wide(r4.l, r2.l, S.L);
  }
}

// The lane's sum of slot q (0..25, the order of the gathered sums) without its
// `fold` lowest bits (room for kFxLanes lanes, no more): the sum is 2^s times
// it with s = fold - kFxBits + a e0 + b e1 + c e2 + d er
template <bool kM6>
FPC_HD int64_t fx_fold(const FxSums<kM6> &S, int q, int fold = kFxFold) {
  if (q < 6) return S.P[q] >> fold;
  const int j = q - 6;
  if (j >= FxSums<kM6>::kN) return 0;
  const int64_t m = j == 19 ? S.M[j] + (S.L >> kFxLimb) : S.M[j];
  return (S.H[j] + (m >> kFxLimb)) >> fold;
}

// a | b << 8 | c << 16 | d << 24 of slot q
FPC_HD uint32_t fx_weights(int q) {
  constexpr uint32_t X = 1u, Y = 1u << 8, Z = 1u << 16, R = 1u << 24;
  const int k = q < 6 ? q : q - 16;  // pair of u_ij, w_ij
  const uint32_t pair = k == 0 ? 2 * X : k == 1 ? X + Y : k == 2 ? X + Z : k == 3 ? 2 * Y : k == 4 ? Y + Z : 2 * Z;
  if (q < 6) return pair;
  if (q < 16) {
    const int t = q - 6;
    return t == 0 ? 3 * X : t == 1 ? 2 * X + Y : t == 2 ? 2 * X + Z : t == 3 ? X + 2 * Y : t == 4 ? X + Y + Z
           : t == 5 ? X + 2 * Z : t == 6 ? 3 * Y : t == 7 ? 2 * Y + Z : t == 8 ? Y + 2 * Z : 3 * Z;
  }
  if (q < 22) return R + pair;
  if (q < 25) return 2 * R + (q == 22 ? X : q == 23 ? Y : Z);
  return 3 * R;
}
FPC_HD int fx_exponent(uint32_t w, const FxCell &c, int fold = kFxFold) {
  return fold - kFxBits + (int)(w & 255u) * c.e[0] + (int)((w >> 8) & 255u) * c.e[1] + (int)((w >> 16) & 255u) * c.e[2] +
         (int)(w >> 24) * c.er;
}

// Whether a cell's tails are too heavy for fixed point: n w_ii > 2^kFxTail u_ii
// max u_jj over the sums.  A Maxwellian has 5 there; one particle far out makes
// it up to n.  Rounding is relative to the largest term that the bounds allow,
// so sums to which ordinary particles contribute beside such a particle (u_12
// beside outliers in c_1 and c_2) lose digits: a thousand particles with
// outliers of 30 to 1e6 sigma came out up to 5,000 times as far off as FP64
// sums, cells below the limit (and those of up to 2^kFxTail particles, which
// cannot pass it) within a few times.
// Compared as logarithms, the doubles' high words (the fraction taken as it is:
// up to 0.09 below); lu: fx_log of u_ii, lmax: the largest of the cell.
constexpr int kFxTail = 4;
FPC_HD int32_t fx_log(uint32_t hi_u, int e, int fold) { return (int32_t)hi_u + (2 * e + fold - kFxBits) * (1 << 20); }
FPC_HD bool fx_heavy(uint32_t hi_w, uint32_t hi_u, uint32_t hi_n, int er, int32_t lmax) {
  return ((int32_t)hi_w - (int32_t)hi_u) + ((int32_t)hi_n - lmax) > (kFxTail - er) * (1 << 20);
}

}  // namespace fpc
