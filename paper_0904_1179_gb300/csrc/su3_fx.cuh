// su3_fx.cuh -- 3x3 complex algebra of FP64 accuracy on the integer and FP32
// pipes of sm_103a.
//
// GB300 has two FP64 lanes per SM and clock (an FP64 FMA occupies an SM for 16
// cycles per warp, measured; so does every conversion to or from FP64), and
// 128 FP32 lanes.  The entries of SU(3) matrices and of their products are
// bounded by 1, so they need no floating exponent: a real is held as
//     x = h 2^-30 + l 2^-62,   h a 32-bit integer, l an FP32 number,
// |l| <= 2^31 nominally (half a unit of h).  A product is
//     x y = hx hy 2^-60 + (hx ly + lx hy) 2^-92 + O(2^-62),
// the first term exact in a 64-bit integer accumulator (one IMAD.WIDE, 1.04
// SM cycles per warp measured), the second in FP32 (two FMAs, 0.72 cycles):
// 1.76 cycles for a multiply-add instead of 16.
//
// Errors are absolute.  l has 24 bits of at most 2^31 units, so a real is held to
// 2^-56 (an FP64 number to 2^-54 where it is between 1/2 and 1, closer below 1/4).
// Sums of the integer part are exact; the cross terms, FP32 sums of up to 2^62 units
// of 2^-92, make an entry of a product of two matrices good to 2^-55 on average and
// 2^-53 at most, as an FP64 FMA chain is at most.  Measured against long double, in
// units of 2^-53, root mean square of a staple's entries here / in FP64
// arithmetic: Haar links 0.94 / 1.50; links eps from the identity, on and off
// the diagonal: eps 0.2 1.08 / 3.90 and 0.96 / 1.15, 0.03 1.14 / 4.59 and 0.94 /
// 0.21, 0.001 1.14 / 4.64 and 0.91 / 0.007, 1e-9 0.04 / 0.21 and 0.48 / 0: small
// entries of nearly ordered configurations are held less closely than by FP64.
// The updated links are not: there FP64 arithmetic loses more in 1 - a0^2 of
// the proposals than a staple's small entries cost here (root mean square off
// the diagonal, GPU, here / FP64: one half-sweep from a cold start at beta 5.7
// 0.37 / 0.80, at 1000 0.32 / 9.6, at 1e6 2.5 / 313; a sweep of a thermal 8 x 6 x
// 4 x 8 lattice at 5.7 0.75 / 1.26, 50 0.61 / 2.7, 5000 0.61 / 27; on the diagonal
// 0.36 to 0.76 / 0.80 to 2.3 in all of them).
//
// Integer sums may wrap on the way (two's complement); only their final value
// has to fit, which the callers' bounds give: entries of near-unitary matrices
// (|x| <= 1 + 2^-9) and of sums of at most six of their products.
#pragma once

#include <cstdint>
#include <cstring>
#include <cmath>
#include <cuda_runtime.h>

namespace su3dev {

#define SU3_HD __host__ __device__ __forceinline__

// FP32 steps with their rounding written out (no contraction left to the
// compiler), so that every kernel that uses them gives the same bits.
SU3_HD float fx_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
SU3_HD float fx_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
SU3_HD float fx_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
SU3_HD float fx_i2f(int a) {
#ifdef __CUDA_ARCH__
  return __int2float_rn(a);
#else
  return (float)a;
#endif
}

// A real: value (h + l 2^-32) unit, f = h rounded to FP32 (the factor of the
// FP32 part of a product).  The unit is 2^-30 unless said otherwise.
struct fx {
  int h;
  float l, f;
};
struct cfx {
  fx re, im;
};
// The same without f (two registers a real, for numbers kept over long code).
struct cfxs {
  int hr, hi;
  float lr, li;
};

SU3_HD fx fx_make(int h, float l) { return fx{h, l, fx_i2f(h)}; }
SU3_HD cfx cfx_of(const cfxs& a) { return cfx{fx_make(a.hr, a.lr), fx_make(a.hi, a.li)}; }
SU3_HD cfxs cfx_short(const cfx& a) { return cfxs{a.re.h, a.im.h, a.re.l, a.im.l}; }
SU3_HD fx fx_neg(fx a) { return fx{-a.h, -a.l, -a.f}; }
SU3_HD cfx cfx_conj(cfx a) { return cfx{a.re, fx_neg(a.im)}; }

// Accumulator of products of units ux, uy: value hh ux uy + c ux uy 2^-32.
struct facc {
  long long hh;
  float c;
};

SU3_HD void fx_mac(facc& s, const fx& a, const fx& b) {
  s.hh += (long long)a.h * b.h;
  s.c = fx_fma(a.f, b.l, s.c);
  s.c = fx_fma(a.l, b.f, s.c);
}
// s - a b (the integer multiplier takes no sign: -a.h is formed once per a)
SU3_HD void fx_msub(facc& s, const fx& a, const fx& b) {
  s.hh += (long long)(-a.h) * b.h;
  s.c = fx_fma(-a.f, b.l, s.c);
  s.c = fx_fma(-a.l, b.f, s.c);
}

// The real of unit u nearest a sum of products in the unit u^2 = u 2^-30: the
// cross terms are added to the integer sum (to 2^-58, F2I on the otherwise idle
// XU), then h = round(hh / 2^30) and l = the remainder.  With l again at most
// half a unit of h the next product's cross terms stay small; carried along as
// they are they made a staple 1.5 times less exact.  2^29 has been added to hh
// (accumulators start from it), which makes the remainder signed.
SU3_HD long long fx_merge(const facc& s) {
#ifdef __CUDA_ARCH__
  const int ci = __float2int_rn(__fmul_rn(s.c, 0x1p-34f));
#else
  const int ci = (int)lrintf(s.c * 0x1p-34f);
#endif
  return s.hh + 4LL * ci;
}
SU3_HD fx fx_norm_merged(long long m) {
  const unsigned long long u = (unsigned long long)m;
  return fx_make((int)(uint32_t)(u >> 30), fx_i2f((int)(((uint32_t)u << 2) + 0x80000000u)));
}
SU3_HD fx fx_norm(const facc& s) { return fx_norm_merged(fx_merge(s)); }
// A merged sum of unit 2^-60 in the unit 2^-28 (the high word; 2^31 added
// before).
SU3_HD fx fx_norm_high(long long m) {
  const unsigned long long u = (unsigned long long)m;
  return fx_make((int)(uint32_t)(u >> 32), fx_i2f((int)((uint32_t)u ^ 0x80000000u)));
}
// Where the accumulator of an fx_norm starts.
SU3_HD facc fx_zero() { return facc{1LL << 29, 0.0f}; }

// An FP64 number with |d| < 2 in units of 2^-62: the mantissa as a 63-bit
// fraction, shifted right by the exponent.  A bit of the value below 2^-62 is
// dropped.  (Integer pipe only: a conversion on the FP64 pipe takes 16 cycles.)
// flip: 0x80000000 negates d.
SU3_HD long long fx_i62_from_double(double d, uint32_t flip = 0u) {
  uint32_t hi, lo;
#ifdef __CUDA_ARCH__
  hi = (uint32_t)__double2hiint(d);
  lo = (uint32_t)__double2loint(d);
#else
  uint64_t b;
  memcpy(&b, &d, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
#endif
  hi ^= flip;
  const uint32_t s = (uint32_t)((int)hi >> 31);
  uint32_t ah = (hi << 10) | (lo >> 22);
  uint32_t al = lo << 10;
  ah = ((ah & 0x3FFFFFFFu) | 0x40000000u) ^ s;  // 1.f as a 63-bit fraction, complemented if negative
  al ^= s;
  // 1023 - exponent, from the complement of the upper word without its sign
  const uint32_t sh = ((~hi | 0x80000000u) >> 20) - (0x800u + 0x7FFu - 1023u);
  const long long m = (long long)(((unsigned long long)ah << 32) | al);
  long long x;
#ifdef __CUDA_ARCH__
  asm("shr.s64 %0, %1, %2;" : "=l"(x) : "l"(m), "r"(sh));  // shifts beyond 63 clamp
#else
  x = m >> (sh > 63 ? 63 : sh);
#endif
  return x;
}
SU3_HD fx fx_from_i62(long long x) {
  const int xl = (int)(uint32_t)x;
  return fx_make((int)(x >> 32) + (int)((uint32_t)xl >> 31), fx_i2f(xl));
}
SU3_HD fx fx_from_double(double d, uint32_t flip = 0u) { return fx_from_i62(fx_i62_from_double(d, flip)); }
// The same by one conversion on the FP64 pipe (busy 40 % of an update's time with these).
SU3_HD fx fx_from_double_cvt(double d, uint32_t flip = 0u) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(d) + (62 << 20);
  return fx_from_i62(__double2ll_rz(__hiloint2double((int)((uint32_t)hi ^ flip), __double2loint(d))));
#else
  return fx_from_double(d, flip);
#endif
}

// The value in units of 2^-62 as a 64-bit integer (l rounded to two of them).
SU3_HD long long fx_to_i64(const fx& a) {
#ifdef __CUDA_ARCH__
  const int li = __float2int_rn(__fmul_rn(a.l, 0.5f));
#else
  const int li = (int)lrintf(a.l * 0.5f);
#endif
  return (long long)a.h * (1LL << 32) + 2LL * li;
}
SU3_HD double fx_to_double(const fx& a) {
  const long long x = fx_to_i64(a);
#ifdef __CUDA_ARCH__
  const double d = __ll2double_rn(x);
  // times 2^-62 on the exponent; zero stays zero
  return x == 0 ? 0.0 : __hiloint2double(__double2hiint(d) - (62 << 20), __double2loint(d));
#else
  return std::ldexp((double)x, -62);
#endif
}

// Complex products into accumulators: s += a b, s += a conj(b) (the host program that measures
// a staple's errors uses this one; the kernels negate as they split), s += conj(a) b.
struct cfacc {
  facc re, im;
};
SU3_HD void cfx_mac(cfacc& s, const cfx& a, const cfx& b) {
  fx_mac(s.re, a.re, b.re);
  fx_msub(s.re, a.im, b.im);
  fx_mac(s.im, a.re, b.im);
  fx_mac(s.im, a.im, b.re);
}
SU3_HD void cfx_mac_cb(cfacc& s, const cfx& a, const cfx& b) {
  fx_mac(s.re, a.re, b.re);
  fx_mac(s.re, a.im, b.im);
  fx_msub(s.im, a.re, b.im);
  fx_mac(s.im, a.im, b.re);
}
SU3_HD void cfx_mac_ca(cfacc& s, const cfx& a, const cfx& b) {
  fx_mac(s.re, a.re, b.re);
  fx_mac(s.re, a.im, b.im);
  fx_mac(s.im, a.re, b.im);
  fx_msub(s.im, a.im, b.re);
}
// s += conj(a b), s -= conj(a b)
SU3_HD void cfx_mac_cc(cfacc& s, const cfx& a, const cfx& b) {
  fx_mac(s.re, a.re, b.re);
  fx_msub(s.re, a.im, b.im);
  fx_msub(s.im, a.re, b.im);
  fx_msub(s.im, a.im, b.re);
}
SU3_HD void cfx_msub_cc(cfacc& s, const cfx& a, const cfx& b) {
  fx_msub(s.re, a.re, b.re);
  fx_mac(s.re, a.im, b.im);
  fx_mac(s.im, a.re, b.im);
  fx_mac(s.im, a.im, b.re);
}
SU3_HD cfacc cfx_zero() { return cfacc{fx_zero(), fx_zero()}; }
SU3_HD cfx cfx_norm(const cfacc& s) { return cfx{fx_norm(s.re), fx_norm(s.im)}; }

// ---------------------------------------------------------------------------
// Staple in this arithmetic: the sum of three-link paths as 64-bit integers in
// units of 2^-60 (at most six paths: 6 2^60 < 2^63).  Integer sums do not depend
// on their order, so lanes that share a link's paths add them up to the same
// bits as one thread does.  Rows 0,1 of a path are the merged sums of its last
// product, row 2 is the merged completion conj(row0 x row1).
// ---------------------------------------------------------------------------
struct fx_rows01 {
  cfx e[2][3];
};
struct fx_staple {
  long long r[3][3][2];
};

SU3_HD void fx_staple_zero(fx_staple& A) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) A.r[i][k][0] = A.r[i][k][1] = 0;
}

// Row 2 of A += F (rows 0,1 given, row 2 completed).  The merged sums of F's rows
// 0,1 (with the 2^29 of fx_zero) are added to A's by who forms them.
SU3_HD void fx_staple_add_row2(fx_staple& A, const fx_rows01& F) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    cfacc s{{A.r[2][k][0], 0.0f}, {A.r[2][k][1], 0.0f}};
    cfx_mac_cc(s, F.e[0][a], F.e[1][b]);
    cfx_msub_cc(s, F.e[0][b], F.e[1][a]);
    A.r[2][k][0] = fx_merge(s.re);
    A.r[2][k][1] = fx_merge(s.im);
  }
}

// One entry of row i of a staple of `paths` paths, in the unit 2^-28 (entries up
// to 6).
SU3_HD fx fx_staple_entry(long long m, int i, int paths) {
  return fx_norm_high(m + ((1LL << 31) - (i < 2 ? (long long)paths << 29 : 0LL)));
}
struct fx_mat {
  cfx e[3][3];
};
SU3_HD fx_mat fx_staple_mat(const fx_staple& A, int paths) {
  fx_mat m;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      m.e[i][k] = cfx{fx_staple_entry(A.r[i][k][0], i, paths), fx_staple_entry(A.r[i][k][1], i, paths)};
  return m;
}

// ---------------------------------------------------------------------------
// Gram-Schmidt of rows 0, 1 of a link that is unitary to within 2^-31 (every
// link is, after rotations of a unitary link): with e = n - 1,
//   r0' = r0 (1 - e0/2),   r1' = (r1 - d r0)(1 - e1/2),   d = <r0, r1>,
// to first order (the second is below 2^-62); the corrections fall in the FP32
// parts.  e and d come from the exact integer sums.  Returns false, with the
// rows unchanged, where a coefficient exceeds 2^-31: the caller takes the
// FP64 Gram-Schmidt.
// ---------------------------------------------------------------------------
// One column's part of |r0|^2, |r1|^2, Re d and Im d, merged; the columns' parts
// add up as integers.
struct fx_gram {
  long long n0, n1, dr, di;
};
SU3_HD fx_gram fx_gram_column(const cfx& a, const cfx& b) {
  facc n0{0, 0.0f}, n1{0, 0.0f};
  cfacc d{{0, 0.0f}, {0, 0.0f}};
  fx_mac(n0, a.re, a.re);
  fx_mac(n0, a.im, a.im);
  fx_mac(n1, b.re, b.re);
  fx_mac(n1, b.im, b.im);
  cfx_mac_ca(d, a, b);
  return fx_gram{fx_merge(n0), fx_merge(n1), fx_merge(d.re), fx_merge(d.im)};
}
// The coefficients of the correction from the whole sums; false where one is
// 2^-31 or more.
struct fx_gs {
  float s0, s1, cr, ci;
};
SU3_HD bool fx_gs_coefficients(const fx_gram& g, fx_gs& c) {
  const long long n0 = g.n0 - (1LL << 60), n1 = g.n1 - (1LL << 60), lim = 1LL << 29;
  const bool ok = n0 < lim && n0 > -lim && n1 < lim && n1 > -lim && g.dr < lim && g.dr > -lim && g.di < lim && g.di > -lim;
  // f is in units of 2^-30, l of 2^-62: a coefficient in units of 2^-60 gets the factor 2^-28
  c.s0 = fx_mul(fx_i2f((int)n0), -0x1p-29f);
  c.s1 = fx_mul(fx_i2f((int)n1), -0x1p-29f);
  c.cr = fx_mul(fx_i2f((int)g.dr), -0x1p-28f);
  c.ci = fx_mul(fx_i2f((int)g.di), -0x1p-28f);
  return ok;
}
SU3_HD void fx_gs_column(const fx_gs& c, cfx& a, cfx& b) {
  b.re.l = fx_fma(c.cr, a.re.f, fx_fma(-c.ci, a.im.f, fx_fma(c.s1, b.re.f, b.re.l)));
  b.im.l = fx_fma(c.cr, a.im.f, fx_fma(c.ci, a.re.f, fx_fma(c.s1, b.im.f, b.im.l)));
  a.re.l = fx_fma(c.s0, a.re.f, a.re.l);
  a.im.l = fx_fma(c.s0, a.im.f, a.im.l);
}

SU3_HD bool fx_reunitarise(fx_mat& u) {
  fx_gram g{0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx_gram q = fx_gram_column(u.e[0][k], u.e[1][k]);
    g.n0 += q.n0;
    g.n1 += q.n1;
    g.dr += q.dr;
    g.di += q.di;
  }
  fx_gs c;
  if (!fx_gs_coefficients(g, c)) return false;
#pragma unroll
  for (int k = 0; k < 3; ++k) fx_gs_column(c, u.e[0][k], u.e[1][k]);
  return true;
}

// Entry k of row 2 of an SU(3) matrix from entries a = k + 1, b = k + 2 (mod 3) of
// rows 0 and 1: conj(x0a x1b - x0b x1a).
SU3_HD cfx fx_row2_entry(const cfx& x0a, const cfx& x0b, const cfx& x1a, const cfx& x1b) {
  cfacc s = cfx_zero();
  cfx_mac_cc(s, x0a, x1b);
  cfx_msub_cc(s, x0b, x1a);
  return cfx_norm(s);
}
SU3_HD void fx_complete_row2(fx_mat& m) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    m.e[2][k] = fx_row2_entry(m.e[0][a], m.e[0][b], m.e[1][a], m.e[1][b]);
  }
}

}  // namespace su3dev
