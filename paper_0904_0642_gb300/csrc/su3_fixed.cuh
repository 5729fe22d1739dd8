// su3_fixed.cuh -- the linear algebra of the FP64 link update in 64-bit fixed
// point.
//
// This GPU executes 2 double-precision FMAs per clock and SM (64 clocks for
// one warp instruction), but 64 wide integer multiply-adds (32 x 32 + 64
// bits).  SU(3) links are bounded by 1, so their products need no exponent:
// a number x is held as the integer x 2^60 in two signed 32-bit limbs,
//   x = (h 2^32 + l) 2^-60,   l in [-2^31, 2^31),
// and a product sum is accumulated exactly in two 64-bit integers,
//   hh = sum h_a h_b          (units 2^-56)
//   x  = sum h_a l_b + l_a h_b (units 2^-88),
// three wide multiply-adds per real product.  The l_a l_b terms are dropped: at
// most 2^-58 each and of either sign, 2^-59.6 root mean square (those of a
// square have one sign: norm_fx adds them).  The result is read as hh 2^32 + x,
// rounded to units 2^-60.  A sum of twelve products is thus within 2^-57.8 root
// mean square (2^-54.4 at most), where each of the double-precision form's
// operations rounds by 2^-54 to 2^-52.
// What goes in and out: elements are read as floor(x 2^60), so that those below
// 2^-7 lose the digits of their doubles beyond 2^-60; links are stored as the
// nearest double; an update's change of Re Tr(U A) is rounded to 2^-51, the last
// place of a double of its size, and a plaquette to 2^-56.
//
// Measured, one update phase: 24^4 (165888 links) 900 us in double, 218 us
// here; 4^4 (128 links) 97 us in double, 32 us here, 11.4 us with eight lanes
// per link.  What bounds it: the integer pipes (53 % of the wide
// multiply-adds' rate and 42 % of the logic's, which share the dispatch, at 8
// warps per SM and 255 registers); 168 and 128 registers (12 and 16 warps per
// SM) are 8 and 16 % slower.
//
// Overflow.  The bounds below hold for any inputs with every element at most
// kElemMax in magnitude (no unitarity assumed), and the results of one stage
// are checked against the same bound before they enter the next:
//   six products (a matrix row times a column): |hh| <= 6.8 2^56, and
//     |x| <= 6 x 2 x 1.0625 x 2^59 = 6.4 2^60 < 2^63;
//   the staple sum: six matrices, 6 x 1.0625 x 2^60 < 2^63;
//   the projection (twelve products of a link and the staple sum, the latter
//     in units 2^-56) folds x into hh after every four.  The rotations of
//     earlier subgroups mix the link's rows and keep their squares' sum, at
//     most 18 x 1.0625^2 = 4.51^2, so that the four elements of a fold add up
//     to 9.02 at most: |x| <= 9.02 2^59 + 4 x 6.4 x 2^55 + 2^32 < 2^63, and
//     |a| <= 4.51 sqrt(2) 15.7 / 2 = 50 (15.7: the norm of a staple column),
//     2^62.7 in units 2^-57;
//   from there on |a| must be below 8 (SU(3) links: at most 6).  norm_fx marks
//     others: they may have no leading zeros left to shift into, and the change
//     of Re Tr(U A) / 2 over the three subgroups, 3 (8 + 8) 2^57 < 2^63, needs
//     the bound too.
// A site that fails a check (links far from SU(3), infinities, NaN) is updated
// by the double-precision form instead.
#pragma once
#include <cstdint>
#include <climits>
#include <cstring>
#include <initializer_list>

#ifdef __CUDACC__
#define SU3_HD __device__ __forceinline__
#define SU3_TABLE static __device__ const
#else
#define SU3_HD inline
#define SU3_TABLE static const
#endif
#include "su3_fixed_tables.h"

namespace su3g {

// The high word of the largest accepted double magnitude (1.0625), and its
// bits as a float.
constexpr uint32_t kElemMaxHi = 0x3FF10000u, kElemMaxFloat = 0x3F880000u;
// The same bound on the high limb (units 2^-28), a margin of one for l < 0.
constexpr int32_t kElemMaxLimb = (17 << 24) + 1;

struct Fx {
  int32_t h, l;
};
struct Fc {
  Fx re, im;
};
struct FM3 {
  Fc e[3][3];
};

SU3_HD int64_t fx_val(const Fx &a) { return (int64_t)a.h * 4294967296ll + a.l; }
SU3_HD Fx fx_split(int64_t v) {
  const uint32_t lo = (uint32_t)v;
  return {(int32_t)((uint32_t)((uint64_t)v >> 32) + (lo >> 31)), (int32_t)lo};
}
// -l of l = -2^31 does not fit a limb: l stays and h takes the carry.
SU3_HD Fx fx_neg(const Fx &a) {
  return {(int32_t)(0u - (uint32_t)a.h + (a.l == INT32_MIN ? 1u : 0u)), (int32_t)(0u - (uint32_t)a.l)};
}

// Range checks, collected over many elements and read once: the largest high
// word of a positive and of a negative double (infinities and NaN included),
// and the extreme high limbs.
struct FxRange {
  int32_t dpos = 0;
  uint32_t dneg = 0;
  int32_t hmax = 0, hmin = 0;
  // high words of doubles, or floats
  SU3_HD void doubles(int32_t hi0, int32_t hi1) {
#ifdef __CUDA_ARCH__
    dpos = __vimax3_s32(dpos, hi0, hi1);
    dneg = __vimax3_u32(dneg, (uint32_t)hi0, (uint32_t)hi1);
#else
    for (const int32_t v : {hi0, hi1}) {
      dpos = v > dpos ? v : dpos;
      dneg = (uint32_t)v > dneg ? (uint32_t)v : dneg;
    }
#endif
  }
  SU3_HD void limbs(int32_t h0, int32_t h1) {
#ifdef __CUDA_ARCH__
    hmax = __vimax3_s32(hmax, h0, h1);
    hmin = __vimin3_s32(hmin, h0, h1);
#else
    for (const int32_t v : {h0, h1}) {
      hmax = v > hmax ? v : hmax;
      hmin = v < hmin ? v : hmin;
    }
#endif
  }
  // top: the high word of the largest accepted double, or its bits as a float
  SU3_HD bool ok(uint32_t top = kElemMaxHi) const {
    return dpos <= (int32_t)top && dneg <= (0x80000000u | top) && hmax <= kElemMaxLimb && hmin >= -kElemMaxLimb;
  }
};

SU3_HD int32_t dbl_hi(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (int32_t)(b >> 32);
#endif
}

SU3_HD uint32_t dbl_lo(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2loint(x);
#else
  int64_t b;
  std::memcpy(&b, &x, 8);
  return (uint32_t)b;
#endif
}
SU3_HD double dbl_make(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
// (hi:lo) >> n for n up to 32, and x >> n with shifts of 32 and more giving 0.
SU3_HD uint32_t shift_r(uint32_t lo, uint32_t hi, uint32_t n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, n);
#else
  return n == 0 ? lo : (n >= 32 ? hi : (lo >> n) | (hi << (32 - n)));
#endif
}
SU3_HD uint32_t shr0(uint32_t x, uint32_t n) {
#ifdef __CUDA_ARCH__
  uint32_t y;
  asm("shr.u32 %0, %1, %2;" : "=r"(y) : "r"(x), "r"(n));
  return y;
#else
  return n > 31 ? 0u : x >> n;
#endif
}
SU3_HD int clz32(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

SU3_HD int clz64(uint64_t x) {
  const uint32_t h = (uint32_t)(x >> 32);
  return h ? clz32(h) : 32 + clz32((uint32_t)x);
}

// v 2^-n rounded to nearest (halves up), 0 <= n < 62.
SU3_HD int64_t shift_round(int64_t v, int n) { return (v + ((1ll << n) >> 1)) >> n; }

// floor(x 2^60) by integer operations, for |x| < 2 (a range check rejects
// others): the mantissa with its leading bit at bit 63, shifted right by
// 1026 - e (zero and subnormals shift out), negative values as the ones'
// complement.
SU3_HD Fx fx_of_mantissa(uint32_t H, uint32_t L, int q, uint32_t s) {
  const int q2 = q > 32 ? q - 32 : 0;
  const uint32_t vh = shr0(H, (uint32_t)q) ^ s;
  const uint32_t vl = shr0(shift_r(L, H, (uint32_t)(q < 32 ? q : 32)), (uint32_t)q2) ^ s;
  return {(int32_t)(vh + (vl >> 31)), (int32_t)vl};
}
SU3_HD Fx fx_of(double x) {
  const uint32_t hi = (uint32_t)dbl_hi(x), lo = dbl_lo(x);
  return fx_of_mantissa((hi << 11 | lo >> 21) | 0x80000000u, lo << 11, 1026 - (int)((hi >> 20) & 0x7FFu),
                        (uint32_t)((int32_t)hi >> 31));
}
// The same for a float.
SU3_HD uint32_t flt_bits(float x) {
  uint32_t u;
#ifdef __CUDA_ARCH__
  u = __float_as_uint(x);
#else
  std::memcpy(&u, &x, 4);
#endif
  return u;
}
SU3_HD Fx fx_of(float x) {
  const uint32_t u = flt_bits(x);
  return fx_of_mantissa((u << 8) | 0x80000000u, 0u, 130 - (int)((u >> 23) & 0xFFu), (uint32_t)((int32_t)u >> 31));
}
// v 2^-60 as a float, rounded to nearest even.
SU3_HD float flt_of(int64_t v) { return (float)v * 0x1p-60f; }
// The same (halves away from zero; zero is not handled), and whether every
// value within 2^12 units (3.6e-15) rounds to it.
SU3_HD float flt_of_sure(int64_t v, bool &sure) {
  const uint64_t m = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
  const int lz = clz64(m);
  const uint64_t n = m << (lz & 63);               // leading bit at 63
  const uint32_t H = (uint32_t)(n >> 32), R = (uint32_t)(n >> 8);  // R: the dropped bits, 2^32 per ulp
  const uint32_t thr = 16u << (lz & 31);
  sure = sure && lz < 27 && R - 0x80000000u + thr > 2u * thr;
  const uint32_t b = (v < 0 ? 0x80000000u : 0u) + ((uint32_t)(127 + 2 - lz) << 23) + (H >> 8) + (R >> 31);
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  std::memcpy(&f, &b, 4);
  return f;
#endif
}

// v 2^-e as a double, rounded to nearest (halves away from zero).
SU3_HD double dbl_of(int64_t v, int e) {
  const uint32_t s = (uint32_t)((uint64_t)v >> 32) & 0x80000000u;
  uint64_t m = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
  const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
  const int lz = mh ? clz32(mh) : 32 + clz32(ml);
  m = (lz < 64 ? m << lz : 0) + 0x400u;  // leading bit at 63; half of the last kept bit
  // a carry out of bit 63 leaves the mantissa zero and steps the exponent
  const uint32_t carry = (uint32_t)(m >> 63) ^ 1u;
  const uint32_t hi = s | (((uint32_t)(1023 + 62 - lz - e + (int)carry) << 20) + ((uint32_t)(m >> 43) | (carry << 20)));
  return v == 0 ? 0.0 : dbl_make(hi, (uint32_t)(m >> 11));
}

// Both by the conversion instructions, which run on the FP64 pipe (16 clocks
// of the SM per warp) beside the integer pipes: faster where many warps wait
// on little else (re-unitarisation of 24^4 FP64 links: 101 -> 81 us), slower
// in the update (225 -> 272 us) and the measurement (296 -> 380 us), whose
// few warps wait for them.
SU3_HD Fx fx_of_pipe(double x) {
#ifdef __CUDA_ARCH__
  return fx_split(__double2ll_rz(dbl_make((uint32_t)dbl_hi(x) + (60u << 20), dbl_lo(x))));
#else
  return fx_of(x);
#endif
}
SU3_HD double dbl_of_pipe(int64_t v, int e) {
  const double d = (double)v;
  return v == 0 ? 0.0 : dbl_make((uint32_t)dbl_hi(d) - ((uint32_t)e << 20), dbl_lo(d));
}

SU3_HD Fc fc_of(double re, double im, FxRange &rg) {
  rg.doubles(dbl_hi(re), dbl_hi(im));
  return {fx_of(re), fx_of(im)};
}

// ------------------------------------------------------------------ product sums

struct FxAcc {
  int64_t hh, x;
};

// One half of 2^-60 in x's units (2^-88): the rounding constant.
constexpr int64_t kHalf60 = 1ll << 27;

SU3_HD void fmac(FxAcc &s, const Fx &a, const Fx &b) {
  s.hh += (int64_t)a.h * b.h;
  s.x += (int64_t)a.h * b.l;
  s.x += (int64_t)a.l * b.h;
}

// The sum in units 2^-56 (the rounding constant added by the caller).
SU3_HD int64_t fold56(const FxAcc &s) {
#ifdef __CUDA_ARCH__
  int64_t v;  // one multiply-add, no sign extension of the high word
  asm("mad.wide.s32 %0, %1, 1, %2;" : "=l"(v) : "r"((int32_t)(s.x >> 32)), "l"(s.hh));
  return v;
#else
  return s.hh + (int64_t)(int32_t)(s.x >> 32);
#endif
}
// The sum in units 2^-60: four more bits from x.
SU3_HD int64_t fold60(const FxAcc &s) {
  const int64_t v = fold56(s);
#ifdef __CUDA_ARCH__
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)((uint64_t)v >> 32);
  return (int64_t)((uint64_t)__funnelshift_l(lo, hi, 4) << 32 | __funnelshift_l((uint32_t)s.x, lo, 4));
#else
  return (int64_t)(((uint64_t)v << 4) | ((uint32_t)s.x >> 28));
#endif
}

// A complex left factor with the one negated part its product needs.
struct FcN {
  Fx re, im, n;
};

// s += a b (n = -a.im)
SU3_HD void cmac_f(FxAcc &re, FxAcc &im, const FcN &a, const Fc &b) {
  fmac(re, a.re, b.re);
  fmac(re, a.n, b.im);
  fmac(im, a.re, b.im);
  fmac(im, a.im, b.re);
}
// s += a conj(b) (n = -a.re)
SU3_HD void cmac_nc_f(FxAcc &re, FxAcc &im, const FcN &a, const Fc &b) {
  fmac(re, a.re, b.re);
  fmac(re, a.im, b.im);
  fmac(im, a.im, b.re);
  fmac(im, a.n, b.im);
}
SU3_HD FcN with_neg_im(const Fc &a) { return {a.re, a.im, fx_neg(a.im)}; }
SU3_HD FcN with_neg_re(const Fc &a) { return {a.re, a.im, fx_neg(a.re)}; }

// p q - r t (the cross product of two rows, not conjugated)
SU3_HD void cross_f(FxAcc &re, FxAcc &im, const Fc &p, const Fx &pim_n, const Fc &q, const Fc &r, const Fx &rre_n,
                    const Fx &rim_n, const Fc &t) {
  fmac(re, p.re, q.re);
  fmac(re, pim_n, q.im);
  fmac(re, rre_n, t.re);
  fmac(re, r.im, t.im);
  fmac(im, p.re, q.im);
  fmac(im, p.im, q.re);
  fmac(im, rre_n, t.im);
  fmac(im, rim_n, t.re);
}

SU3_HD void store60(Fc &c, const FxAcc &re, const FxAcc &im, FxRange &rg) {
  c = {fx_split(fold60(re)), fx_split(fold60(im))};
  rg.limbs(c.re.h, c.im.h);
}

// Third row of an SU(3) matrix from rows 0, 1: conj(row 0 x row 1).
SU3_HD void third_row_f(FM3 &m, FxRange &rg) {
  Fx nr[3], ni[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    nr[j] = fx_neg(m.e[0][j].re);
    ni[j] = fx_neg(m.e[0][j].im);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int p = (j + 1) % 3, r = (j + 2) % 3;
    FxAcc re = {0, kHalf60}, im = {0, kHalf60};
    cross_f(re, im, m.e[0][p], ni[p], m.e[1][r], m.e[0][r], nr[r], ni[r], m.e[1][p]);
    const int64_t vi = fold60(im);
    m.e[2][j] = {fx_split(fold60(re)), fx_split(-vi)};
    rg.limbs(m.e[2][j].re.h, m.e[2][j].im.h);
  }
}

// The staple sum in units 2^-60.
struct FSum {
  int64_t re[3][3], im[3][3];
};

// A += m for an SU(3) matrix m given by rows 0, 1 (its third row from the
// cross product, as in the double-precision form).
SU3_HD void acc_su3_2rows_f(FSum &A, const FM3 &m, FxRange &rg) {
  FM3 full = m;
  third_row_f(full, rg);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      A.re[i][j] += fx_val(full.e[i][j].re);
      A.im[i][j] += fx_val(full.e[i][j].im);
    }
}

// Row i of a b: row i of a given.
SU3_HD void row_nn_f(FM3 &c, int i, const Fc (&a)[3], const FM3 &b, FxRange &rg) {
  const FcN l[3] = {with_neg_im(a[0]), with_neg_im(a[1]), with_neg_im(a[2])};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxAcc re = {0, kHalf60}, im = {0, kHalf60};
#pragma unroll
    for (int k = 0; k < 3; ++k) cmac_f(re, im, l[k], b.e[k][j]);
    store60(c.e[i][j], re, im, rg);
  }
}

// Row i of a b^+: row i of a given.
SU3_HD void row_nd_f(FM3 &c, int i, const Fc (&a)[3], const FM3 &b, FxRange &rg) {
  const FcN l[3] = {with_neg_re(a[0]), with_neg_re(a[1]), with_neg_re(a[2])};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    FxAcc re = {0, kHalf60}, im = {0, kHalf60};
#pragma unroll
    for (int k = 0; k < 3; ++k) cmac_nc_f(re, im, l[k], b.e[j][k]);
    store60(c.e[i][j], re, im, rg);
  }
}

SU3_HD Fx fx_sel(bool c, const Fx &a, const Fx &b) { return {c ? a.h : b.h, c ? a.l : b.l}; }
SU3_HD Fc fc_sel(bool c, const Fc &a, const Fc &b) { return {fx_sel(c, a.re, b.re), fx_sel(c, a.im, b.im)}; }

// One staple added to A.  With M = X Y (rows 0, 1 of X given):
//   upper (up): G M^+ = a (c b)^+, X = U_nu(x), Y = U_mu(x+nu), G = U_nu(x+mu);
//   lower: M^+ G = (e f)^+ h, X = U_mu(x-nu), Y = U_nu(x+mu-nu), G = U_nu(x-nu).
// Both through one sequence of instructions, M^+ G = conj(M^T conj(G^T)^T):
// sites and lanes of both kinds run together, and the code is half as long.
SU3_HD void staple_f(FSum &A, const Fc (&X)[2][3], const FM3 &Y, const FM3 &G, bool up, FxRange &rg) {
  FM3 M, P;
#pragma unroll
  for (int i = 0; i < 2; ++i) row_nn_f(M, i, X[i], Y, rg);
  third_row_f(M, rg);
  FM3 B;
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < 3; ++k) B.e[j][k] = fc_sel(up, M.e[j][k], G.e[k][j]);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    Fc l[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) l[k] = fc_sel(up, G.e[i][k], M.e[k][i]);
    row_nd_f(P, i, l, B, rg);
#pragma unroll
    for (int k = 0; k < 3; ++k) P.e[i][k].im = fx_sel(up, P.e[i][k].im, fx_neg(P.e[i][k].im));
  }
  acc_su3_2rows_f(A, P, rg);
}

// Re Tr(P Q^+) of two SU(3) matrices given by rows 0, 1 (plaquette_at in
// su3_site.cuh), in units 2^-60.
SU3_HD int64_t trace_nd_f(const FM3 &P, const FM3 &Q, FxRange &rg) {
  Fc G[2][2];  // <P_k, Q_l>
#pragma unroll
  for (int l = 0; l < 2; ++l) {
    const FcN q[3] = {with_neg_re(Q.e[l][0]), with_neg_re(Q.e[l][1]), with_neg_re(Q.e[l][2])};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      FxAcc re = {0, kHalf60}, im = {0, kHalf60};
#pragma unroll
      for (int j = 0; j < 3; ++j) cmac_nc_f(re, im, q[j], P.e[k][j]);
      store60(G[k][l], re, im, rg);
    }
  }
  FxAcc t = {0, kHalf60};
  fmac(t, G[0][0].re, G[1][1].re);
  fmac(t, fx_neg(G[0][0].im), G[1][1].im);
  fmac(t, fx_neg(G[0][1].re), G[1][0].re);
  fmac(t, G[0][1].im, G[1][0].im);
  return fold60(t) + fx_val(G[0][0].re) + fx_val(G[1][1].re);
}

// The staple sum as a factor: units 2^-56, so that the twelve products of a
// projection stay inside 64 bits.
SU3_HD FM3 factor56(const FSum &A) {
  FM3 m;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) m.e[i][j] = {fx_split((A.re[i][j] + 8) >> 4), fx_split((A.im[i][j] + 8) >> 4)};
  return m;
}

// ------------------------------------------------------------------ Cabibbo-Marinari

// The quaternion projection of the (i, j) block of U A (block_projection in
// su3_device.cuh), U in units 2^-60 and A in units 2^-56: four sums over k of
// four products of u_ik, u_jk, a_ki, a_kj.  One k:
SU3_HD void project_k_f(FxAcc (&s)[4], const Fc &ui, const Fc &uj, const Fc &ai, const Fc &aj) {
  const Fx ni = fx_neg(ui.im), nre = fx_neg(uj.re), nim = fx_neg(uj.im);
  // Re(u_ik a_ki + u_jk a_kj)
  fmac(s[0], ui.re, ai.re);
  fmac(s[0], ni, ai.im);
  fmac(s[0], uj.re, aj.re);
  fmac(s[0], nim, aj.im);
  // Im(u_ik a_kj + u_jk a_ki)
  fmac(s[1], ui.re, aj.im);
  fmac(s[1], ui.im, aj.re);
  fmac(s[1], uj.re, ai.im);
  fmac(s[1], uj.im, ai.re);
  // Re(u_ik a_kj - u_jk a_ki)
  fmac(s[2], ui.re, aj.re);
  fmac(s[2], ni, aj.im);
  fmac(s[2], nre, ai.re);
  fmac(s[2], uj.im, ai.im);
  // Im(u_ik a_ki - u_jk a_kj)
  fmac(s[3], ui.re, ai.im);
  fmac(s[3], ui.im, ai.re);
  fmac(s[3], nre, aj.im);
  fmac(s[3], nim, aj.re);
#pragma unroll
  for (int q = 0; q < 4; ++q) s[q] = {fold56(s[q]), (int64_t)(uint32_t)s[q].x};  // the same sum, x below 2^32
}

// rotate_rows of one column of rows i, j by the unit quaternion r (n: its
// negated vector part).
SU3_HD void rotate_col_f(Fc &ui, Fc &uj, const Fx (&r)[4], const Fx (&n)[4]) {
  const Fc a = ui, b = uj;
  FxAcc s[4] = {{0, kHalf60}, {0, kHalf60}, {0, kHalf60}, {0, kHalf60}};
  fmac(s[0], r[0], a.re);
  fmac(s[0], n[3], a.im);
  fmac(s[0], r[2], b.re);
  fmac(s[0], n[1], b.im);
  fmac(s[1], r[0], a.im);
  fmac(s[1], r[3], a.re);
  fmac(s[1], r[2], b.im);
  fmac(s[1], r[1], b.re);
  fmac(s[2], n[2], a.re);
  fmac(s[2], n[1], a.im);
  fmac(s[2], r[0], b.re);
  fmac(s[2], r[3], b.im);
  fmac(s[3], n[2], a.im);
  fmac(s[3], r[1], a.re);
  fmac(s[3], r[0], b.im);
  fmac(s[3], n[3], b.re);
  ui = {fx_split(fold60(s[0])), fx_split(fold60(s[1]))};
  uj = {fx_split(fold60(s[2])), fx_split(fold60(s[3]))};
}

// ------------------------------------------------------------------ functions of the draw
// The logarithm, sine, cosine and reciprocal square root of the heatbath's
// draw, from the 32-bit random words, in the same integers: table steps and
// Taylor series, absolute errors below 2^-56 (measured against quadruple
// precision over 10^7 words: logarithm 0.9, sine and cosine 4, reciprocal
// square root 8 units of 2^-60).

// a b in units 2^-60 (of a in 2^-60 and b in 2^-60; other units scale along).
SU3_HD int64_t fx_mul(const Fx &a, const Fx &b) {
  FxAcc s = {0, kHalf60};
  fmac(s, a, b);
  return fold60(s);
}

// -ln((w + 1/2) / 2^32) in units 2^-57.  With N = 2 w + 1 = 2^(32 - z) m,
// m in [1, 2), and c from the table so that r = m c - 1 is exact and |r| <
// 0.0043: z ln 2 + (ln 2 + ln c) - ln(1 + r).
SU3_HD int64_t neg_log_fx(uint32_t w) {
  const int z = clz32(w);
  const uint32_t m = z > 31 ? 0u : (2u * w + 1u) << z;  // the 32 bits after the leading one
  const TabEntry t = kLogTab[m >> 25];
  const uint32_t c = (uint32_t)t.a;
  const int64_t r60 = ((int64_t)((uint64_t)m * c + ((uint64_t)c << 32)) - (1ll << 42)) * (1 << 18);
  const int32_t r = (int32_t)(r60 >> 22);  // units 2^-38
  // ln(1 + r) = r - r^2 (1/2 - r (1/3 - r (1/4 - r (1/5 - r (1/6 - r / 7)))))
  const int32_t w5 = 1431655765 - (int32_t)(((int64_t)r * 19173961) >> 32);  // 2^-33
  const int32_t w4 = 1717986918 - (int32_t)(((int64_t)r * w5) >> 38);        // 2^-33
  const int32_t w3 = (1 << 30) - (int32_t)(((int64_t)r * w4) >> 39);         // 2^-32
  const int32_t w2 = 1431655765 - (int32_t)(((int64_t)r * w3) >> 38);        // 2^-32
  const Fx rf = fx_split(r60);
  const int64_t q = (1ll << 59) - (((int64_t)r * w2) >> 10);                 // 2^-60
  const int64_t ln1p = r60 - fx_mul(rf, fx_split(fx_mul(rf, fx_split(q))));
  return z * kLn2_57 + ((t.b - ln1p + 4) >> 3);
}

// cos and sin of 2 pi (w + half / 2) / 2^32 (half 0 or 1) in units 2^-60: the
// nearest of 128 angles from the table and the rest, |d| < pi / 128.
SU3_HD void trig_fx(uint32_t w, int half, int64_t &cs, int64_t &sn) {
  const uint32_t t = w + (1u << 24);
  const TabEntry e = kTrigTab[t >> 25];
  const int32_t d = 2 * ((int32_t)(t & 0x1FFFFFFu) - (1 << 24)) + half;  // 2^-33 turns
  // d 2 pi 2^27 = d kTwoPi_59 / 2^32
  const Fx k = fx_split(kTwoPi_59);
  const Fx df = fx_split((int64_t)d * k.h + (((int64_t)d * k.l + (1ll << 31)) >> 32));
  const int64_t d2 = fx_mul(df, df);
  const Fx d2f = fx_split(d2);
  const int32_t D = (int32_t)((d2 + (1 << 18)) >> 19);  // units 2^-41
  // cos d = 1 - d^2 (1/2 - d^2 (1/24 - d^2 / 720))
  const int32_t c2 = 1431655765 - (int32_t)(((int64_t)D * 93207) >> 32);  // 2^-35
  const int64_t c1 = (1ll << 59) - (((int64_t)D * c2) >> 16);
  const Fx cd = fx_split((1ll << 60) - fx_mul(d2f, fx_split(c1)));
  // sin d = d (1 - d^2 (1/6 - d^2 (1/120 - d^2 / 5040)))
  const int32_t s3 = 1145324612 - (int32_t)(((int64_t)D * 53261) >> 32);  // 2^-37
  const int64_t s2 = 192153584101141163ll - (((int64_t)D * s3) >> 18);
  const Fx sd = fx_split(fx_mul(df, fx_split((1ll << 60) - fx_mul(d2f, fx_split(s2)))));
  const Fx ec = fx_split(e.a), es = fx_split(e.b);
  FxAcc a = {0, kHalf60};
  fmac(a, ec, cd);
  fmac(a, fx_split(-e.b), sd);
  cs = fold60(a);
  FxAcc b = {0, kHalf60};
  fmac(b, es, cd);
  fmac(b, ec, sd);
  sn = fold60(b);
}

SU3_HD float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}

// 1 / sqrt(n), n in [1/4, 4) (units 2^-60 both): a float seed Y (2^-26) and
// one third-order step, y (1 + e/2 + 3 e^2 / 8) with e = 1 - n y^2, |e| < 2^-20.
SU3_HD int64_t rsqrt_fx(const Fx &n) {
  const int32_t Y = (int32_t)(rsqrt_seed((float)n.h * 0x1p-28f) * 0x1p26f);
  const auto mulY = [Y](const Fx &a) { return ((int64_t)a.h * Y) * 64 + (((int64_t)a.l * Y) >> 26); };
  const int64_t e = (1ll << 60) - mulY(fx_split(mulY(n)));
  const int32_t es = (int32_t)(e >> 12);  // 2^-48
  const int64_t g = (e >> 1) + ((3 * (((int64_t)es * es) >> 36)) >> 3);
  return ((int64_t)Y << 34) + mulY(fx_split(g));
}

// sqrt(p), p > 0 in units 2^-64: the result times 2^e, in [1/2, 1) and in
// units 2^-60.
SU3_HD int64_t sqrt_u64(uint64_t p, int &e) {
  const int z = clz64(p) & ~1;
  const Fx n = fx_split((int64_t)((p << z) >> 4));  // [1/4, 1)
  e = z >> 1;
  return fx_mul(n, fx_split(rsqrt_fx(n)));
}

// ------------------------------------------------------------------ re-unitarisation
// Gram-Schmidt of rows 0, 1; false when a squared norm leaves [1/4, 4).

SU3_HD int64_t norm2_f(const Fc (&a)[3]) {
  FxAcc n = {0, kHalf60};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    fmac(n, a[k].re, a[k].re);
    fmac(n, a[k].im, a[k].im);
  }
  return fold60(n);
}
SU3_HD bool norm2_ok(int64_t n) { return n >= (1ll << 58) && n < (1ll << 62); }

// q = sum_k conj(a_k) b_k
SU3_HD void inner_f(const Fc (&a)[3], const Fc (&b)[3], int64_t &qr, int64_t &qi) {
  FxAcc re = {0, kHalf60}, im = {0, kHalf60};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    fmac(re, a[k].re, b[k].re);
    fmac(re, a[k].im, b[k].im);
    fmac(im, a[k].re, b[k].im);
    fmac(im, fx_neg(a[k].im), b[k].re);
  }
  qr = fold60(re);
  qi = fold60(im);
}

// n^(-1/2): to rounding level (FLOAT = false), or as the double-precision form
// takes it for float storage - a float seed and one Newton step, exact to
// ~1e-13 - so that the stored floats are that form's.
template <bool FLOAT>
SU3_HD int64_t reunit_rsqrt_fx(int64_t n) {
  const Fx nf = fx_split(n);
  if (!FLOAT) return rsqrt_fx(nf);
  const int64_t y = fx_val(fx_of(rsqrt_seed(flt_of(n))));
  const Fx yf = fx_split(y);
  const int64_t e = (1ll << 60) - fx_mul(fx_split(fx_mul(nf, yf)), yf);  // 1 - n y^2
  return y + fx_mul(fx_split(e >> 1), yf);
}

template <bool FLOAT>
SU3_HD bool reunit_f(FM3 &m, FxRange &rg) {
  Fc(&a)[3] = m.e[0], (&b)[3] = m.e[1];
  const int64_t n1 = norm2_f(a);
  if (!norm2_ok(n1)) return false;
  const Fx s1 = fx_split(reunit_rsqrt_fx<FLOAT>(n1));
#pragma unroll
  for (int k = 0; k < 3; ++k) a[k] = {fx_split(fx_mul(a[k].re, s1)), fx_split(fx_mul(a[k].im, s1))};
  int64_t qr, qi;
  inner_f(a, b, qr, qi);
  const Fx pr = fx_split(-qr), pi = fx_split(-qi), pn = fx_split(qi);
#pragma unroll
  for (int k = 0; k < 3; ++k) {  // b - q a
    FxAcc re = {0, kHalf60}, im = {0, kHalf60};
    fmac(re, pr, a[k].re);
    fmac(re, pn, a[k].im);
    fmac(im, pr, a[k].im);
    fmac(im, pi, a[k].re);
    b[k] = {fx_split(fx_val(b[k].re) + fold60(re)), fx_split(fx_val(b[k].im) + fold60(im))};
  }
  const int64_t n2 = norm2_f(b);
  if (!norm2_ok(n2)) return false;
  const Fx s2 = fx_split(reunit_rsqrt_fx<FLOAT>(n2));
#pragma unroll
  for (int k = 0; k < 3; ++k) b[k] = {fx_split(fx_mul(b[k].re, s2)), fx_split(fx_mul(b[k].im, s2))};
  third_row_f(m, rg);
  return true;
}

// The factors of reunit_rows2_f (su3_site.cuh) from two float rows: e1 = s1 -
// 1, p = s1 <r1, r2>, e2 = s2 - 1 with s1 = n1^(-1/2), s2 = (n2 - |p|^2)^(-1/2).
SU3_HD bool reunit_factors_f(const Fc (&a)[3], const Fc (&b)[3], float &e1, float &pr, float &pi, float &e2) {
  const int64_t n1 = norm2_f(a);
  if (!norm2_ok(n1)) return false;
  const int64_t s1 = reunit_rsqrt_fx<true>(n1);
  int64_t qr, qi;
  inner_f(a, b, qr, qi);
  const Fx s1f = fx_split(s1);
  const int64_t vr = fx_mul(fx_split(qr), s1f), vi = fx_mul(fx_split(qi), s1f);
  FxAcc p2 = {0, kHalf60};
  const Fx fr = fx_split(vr), fi = fx_split(vi);
  fmac(p2, fr, fr);
  fmac(p2, fi, fi);
  const int64_t n2 = norm2_f(b) - fold60(p2);
  if (!norm2_ok(n2)) return false;
  const int64_t s2 = reunit_rsqrt_fx<true>(n2);
  e1 = flt_of(s1 - (1ll << 60));
  pr = flt_of(vr);
  pi = flt_of(vi);
  e2 = flt_of(s2 - (1ll << 60));
  return true;
}

// ------------------------------------------------------------------ the draw

// 3 / (2 beta) = m 2^e, m in [1/2, 1) in units 2^-60 (beta = 0: e huge).
struct InvBeta {
  int64_t m;
  int32_t e;
};

// |a| of a projection: a[q] (units 2^-57) = v[q] k with v a unit quaternion.
// k = kappa 2^(3 - s), kappa and its inverse y in units 2^-60, s >= 0.
struct FxNorm {
  Fx v[4];
  Fx y;
  int64_t kappa;
  int s;
};

// false when a vanishes or has a component of 8 or more; large becomes negative
// when the norm is 8 or more.  The callers read it once, after the three
// subgroups: no branch waits for kappa (one that did cost 1 %).  KEEP: only
// the sign changes, and a count of proposals can carry it (a register of its
// own costs the one-thread update 1 %, the masks the eight-lane one).
template <bool KEEP>
SU3_HD bool norm_fx(const int64_t a[4], FxNorm &n, int32_t &large) {
  constexpr int32_t kMask = KEEP ? INT32_MIN : -1;
  uint64_t top = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) top |= (uint64_t)(a[q] ^ (a[q] >> 63));
  const int s = clz64(top) - 4;  // the largest |a| to [1/2, 1)
  large |= s & kMask;
  if ((uint32_t)s > 59u) return false;  // a = 0: s = 60
  FxAcc sum = {0, kHalf60};
  Fx f[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    f[q] = fx_split(a[q] << s);
    fmac(sum, f[q], f[q]);
    // the product that fmac drops has one sign here: without it the norm is
    // low by 4 units on average, and the booked action drifts
    sum.x += ((int64_t)f[q].l * f[q].l) >> 32;
  }
  const Fx n2 = fx_split(fold60(sum));
  n.y = fx_split(rsqrt_fx(n2));
  n.kappa = fx_mul(n2, n.y);
#pragma unroll
  for (int q = 0; q < 4; ++q) n.v[q] = fx_split(fx_mul(f[q], n.y));
  n.s = s;
  if (s == 0) large |= (int32_t)((uint32_t)((uint64_t)n.kappa >> 32) << 3) & kMask;  // kappa < 2: 1 is the sign bit
  return true;
}

// X = L / alpha of one Kennedy-Pendleton proposal as Q 2^e (Q in units 2^-60,
// [1/8, 2)) and in units 2^-60.
struct Proposal {
  int64_t Q, X;
  int e;
};
enum ProposalStatus { kRejected = 0, kAccepted = 1, kInDouble = 2 };

// L = -(ln u1 + cos^2(2 pi u2) ln u3) in units 2^-57 (< 46) from the two
// logarithms and cs = cos(4 pi u2).
SU3_HD int64_t radius_fx(int64_t nl1, int64_t nl3, int64_t cs) {
  return nl1 + fx_mul(fx_split(nl3), fx_split(((1ll << 60) + cs) >> 1));
}

// u4^2 in units 2^-60, u4 = (2 w + 1) / 2^33: w (w + 1) / 2^4 (+ 2^-6).
SU3_HD int64_t square_fx(uint32_t w) { return (int64_t)(((uint64_t)w * w + w) >> 4); }

// One proposal: 1 / alpha = y 2^(s - 3) 3 / (2 beta), accepted when u4^2 <=
// 1 - X / 2.  L below 2^-12 (five draws in a million) has too few digits
// here: such a draw is left to the double-precision form.
SU3_HD ProposalStatus propose_fx(int64_t L, int64_t u4sq, const FxNorm &n, const InvBeta &ib, Proposal &p) {
  if (L < (1ll << 45)) return kInDouble;
  const int z = clz64((uint64_t)L) - 4;  // to [1/2, 1)
  const Fx Ln = fx_split(z >= 0 ? L << z : L >> -z);
  p.Q = fx_mul(fx_split(fx_mul(Ln, n.y)), fx_split(ib.m));
  p.e = ib.e + n.s - z;
  const int e = p.e;
  if (e > 4) return kRejected;  // X >= 2
  if (e > 0 && (p.Q >> (61 - e)) != 0) return kRejected;
  p.X = e >= 0 ? p.Q << e : (e > -64 ? p.Q >> -e : 0);
  if (p.X >= (1ll << 61)) return kRejected;
  return u4sq <= (1ll << 60) - (p.X >> 1) ? kAccepted : kRejected;
}

// The direction's parts from its two words.
struct Direction {
  Fx st, ct, cphi, sphi;  // sin, cos of theta and phi
};
SU3_HD Fx cos_theta_fx(uint32_t w) { return fx_split(((int64_t)w * 2 + 1 - (1ll << 32)) * (1 << 28)); }
// sin(theta) = 2 sqrt(u (1 - u)): (2 w + 1) (2^33 - 2 w - 1) = 4 w ~w + 2^33 - 1
SU3_HD Fx sin_theta_fx(uint32_t w) {
  int e;
  const int64_t s = sqrt_u64(((uint64_t)w * (uint32_t)~w << 2) + 0x1FFFFFFFFull, e);
  return fx_split(s >> e);
}

// x = (1 - X, isotropic of length sqrt(X (2 - X))).
SU3_HD void direction_fx(const Proposal &p, const Direction &dir, Fx (&x)[4]) {
  // X (2 - X) = P 2^e, e even
  int64_t P = fx_mul(fx_split(p.Q), fx_split((1ll << 61) - p.X));
  P = (P << (p.e & 1)) | 1;
  int ze;
  const int64_t sq = sqrt_u64((uint64_t)P, ze);  // sqrt(P) / 4 = sq 2^-ze
  const int sh = ze - 2 - (p.e >> 1);            // the length is at most 1: sh >= 0
  const Fx rho = fx_split(sq >> (sh < 0 ? 0 : (sh > 63 ? 63 : sh)));
  const Fx t = fx_split(fx_mul(rho, dir.st));
  x[0] = fx_split((1ll << 60) - p.X);
  x[1] = fx_split(fx_mul(t, dir.cphi));
  x[2] = fx_split(fx_mul(t, dir.sphi));
  x[3] = fx_split(fx_mul(rho, dir.ct));
}

// r = x v^+ as quaternions.
SU3_HD void quat_fx(const Fx (&x)[4], const Fx (&v)[4], Fx (&r)[4]) {
  const Fx n1 = fx_neg(x[1]), n2 = fx_neg(x[2]), n3 = fx_neg(x[3]), n0 = fx_neg(x[0]);
  FxAcc s[4] = {{0, kHalf60}, {0, kHalf60}, {0, kHalf60}, {0, kHalf60}};
#pragma unroll
  for (int q = 0; q < 4; ++q) fmac(s[0], x[q], v[q]);
  fmac(s[1], n0, v[1]);
  fmac(s[1], x[1], v[0]);
  fmac(s[1], x[2], v[3]);
  fmac(s[1], n3, v[2]);
  fmac(s[2], n0, v[2]);
  fmac(s[2], x[2], v[0]);
  fmac(s[2], x[3], v[1]);
  fmac(s[2], n1, v[3]);
  fmac(s[3], n0, v[3]);
  fmac(s[3], x[3], v[0]);
  fmac(s[3], x[1], v[2]);
  fmac(s[3], n2, v[1]);
#pragma unroll
  for (int q = 0; q < 4; ++q) r[q] = fx_split(fold60(s[q]));
}

}  // namespace su3g
