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
// 1.76 cycles for a multiply-add instead of 16.  Sums of the integer part are
// exact; the FP32 part is 2^-31 of the result, so its rounding errors are
// about 2^-57 of a matrix entry -- below the 2^-54 of FP64 arithmetic, which
// rounds every partial sum.
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

SU3_HD fx fx_make(int h, float l) { return fx{h, l, fx_i2f(h)}; }
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
SU3_HD fx fx_norm(const facc& s) {
  const unsigned long long u = (unsigned long long)fx_merge(s);
  return fx_make((int)(uint32_t)(u >> 30), fx_i2f((int)(((uint32_t)u << 2) + 0x80000000u)));
}
// Sums of reals (not of products): h = round(hh / 4), for the unit 4 u.
SU3_HD fx fx_norm_sum(const facc& s) {
  const unsigned long long u = (unsigned long long)s.hh;
  const int rem = (int)(((uint32_t)u << 30) + 0x80000000u);
  return fx_make((int)(uint32_t)(u >> 2), fx_fma(s.c, 0.25f, fx_i2f(rem)));
}
// A merged sum of unit 2^-60 in the unit 2^-28 (the high word; 2^31 added
// before).
SU3_HD fx fx_norm_high(const facc& s) {
  const unsigned long long u = (unsigned long long)s.hh;
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
// The same by one conversion on the FP64 pipe, which is otherwise idle.
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

// Complex products into accumulators: s += a b, s += a conj(b), s += conj(a) b.
struct cfacc {
  facc re, im;
};
SU3_HD void cfx_mac(cfacc& s, const cfx& a, const cfx& b) {
  fx_mac(s.re, a.re, b.re);
  fx_msub(s.re, a.im, b.im);
  fx_mac(s.im, a.re, b.im);
  fx_mac(s.im, a.im, b.re);
}
SU3_HD void cfx_msub(cfacc& s, const cfx& a, const cfx& b) {
  fx_msub(s.re, a.re, b.re);
  fx_mac(s.re, a.im, b.im);
  fx_msub(s.im, a.re, b.im);
  fx_msub(s.im, a.im, b.re);
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
SU3_HD cfx cfx_norm_high(const cfacc& s) { return cfx{fx_norm_high(s.re), fx_norm_high(s.im)}; }

// ---------------------------------------------------------------------------
// Staple in this arithmetic.  A three-link path's rows 0,1 come out in the unit
// 2^-30.  The staple's rows 0,1 are sums of at most six of them: the h summed
// in 64 bits, the l in FP32; its row 2 is accumulated from the completions
// conj(row0 x row1) in the unit 2^-60.
// ---------------------------------------------------------------------------
struct fx_rows01 {
  cfx e[2][3];
};
struct fx_staple {
  facc r01[2][3][2];  // sums of h and l (rows 0, 1; re, im)
  cfacc r2[3];          // merged
};

SU3_HD void fx_staple_zero(fx_staple& A) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int c = 0; c < 2; ++c) A.r01[i][k][c] = facc{2, 0.0f};
#pragma unroll
  for (int k = 0; k < 3; ++k) A.r2[k] = cfacc{{1LL << 31, 0.0f}, {1LL << 31, 0.0f}};
}

// A += F (rows 0,1 given, row 2 completed).
SU3_HD void fx_staple_add(fx_staple& A, const fx_rows01& F) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      A.r01[i][k][0].hh += F.e[i][k].re.h;
      A.r01[i][k][1].hh += F.e[i][k].im.h;
      A.r01[i][k][0].c = fx_add(A.r01[i][k][0].c, F.e[i][k].re.l);
      A.r01[i][k][1].c = fx_add(A.r01[i][k][1].c, F.e[i][k].im.l);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    // the cross terms path by path: six paths' in one FP32 sum lose up to three bits
    cfacc s{{A.r2[k].re.hh, 0.0f}, {A.r2[k].im.hh, 0.0f}};
    cfx_mac_cc(s, F.e[0][a], F.e[1][b]);
    cfx_msub_cc(s, F.e[0][b], F.e[1][a]);
    A.r2[k].re.hh = fx_merge(s.re);
    A.r2[k].im.hh = fx_merge(s.im);
  }
}

// The staple as a matrix in the unit 2^-28 (entries up to 6).
struct fx_mat {
  cfx e[3][3];
};
SU3_HD fx_mat fx_staple_mat(const fx_staple& A) {
  fx_mat m;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m.e[i][k].re = fx_norm_sum(A.r01[i][k][0]);
      m.e[i][k].im = fx_norm_sum(A.r01[i][k][1]);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) m.e[2][k] = cfx_norm_high(A.r2[k]);
  return m;
}

// Row 2 of an SU(3) matrix (unit 2^-30) from rows 0 and 1: conj(row0 x row1).
SU3_HD void fx_complete_row2(fx_mat& m) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    cfacc s = cfx_zero();
    cfx_mac_cc(s, m.e[0][a], m.e[1][b]);
    cfx_msub_cc(s, m.e[0][b], m.e[1][a]);
    m.e[2][k] = cfx_norm(s);
  }
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
// A small sum in units of 2^-60 as FP32 (ok = false where it is not small):
// its integer part reaches 2.5 2^30 (cancelled by the FP32 part, the cross
// terms of h and l), so it is taken without its last four bits.
SU3_HD float fx_small(const facc& s, bool& ok) {
  const float v = fx_fma(fx_i2f((int)(s.hh >> 4)), 16.0f, fx_mul(s.c, 0x1p-32f));
  ok = ok && s.hh < (1LL << 34) && s.hh > -(1LL << 34) && v < 0x1p29f && v > -0x1p29f;
  return v;
}

SU3_HD bool fx_reunitarise(fx_mat& u) {
  // half of the four bits that fx_small drops
  facc n0{8 - (1LL << 60), 0.0f}, n1 = n0;
  cfacc d{{8, 0.0f}, {8, 0.0f}};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    fx_mac(n0, u.e[0][k].re, u.e[0][k].re);
    fx_mac(n0, u.e[0][k].im, u.e[0][k].im);
    fx_mac(n1, u.e[1][k].re, u.e[1][k].re);
    fx_mac(n1, u.e[1][k].im, u.e[1][k].im);
    cfx_mac_ca(d, u.e[0][k], u.e[1][k]);
  }
  bool ok = true;
  const float e0 = fx_small(n0, ok), e1 = fx_small(n1, ok), dr = fx_small(d.re, ok), di = fx_small(d.im, ok);
  if (!ok) return false;
  // f is in units of 2^-30, l of 2^-62: a coefficient in units of 2^-60 gets the factor 2^-28
  const float s0 = fx_mul(e0, -0x1p-29f), s1 = fx_mul(e1, -0x1p-29f);
  const float cr = fx_mul(dr, -0x1p-28f), ci = fx_mul(di, -0x1p-28f);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cfx& a = u.e[0][k];
    cfx& b = u.e[1][k];
    b.re.l = fx_fma(cr, a.re.f, fx_fma(-ci, a.im.f, fx_fma(s1, b.re.f, b.re.l)));
    b.im.l = fx_fma(cr, a.im.f, fx_fma(ci, a.re.f, fx_fma(s1, b.im.f, b.im.l)));
    a.re.l = fx_fma(s0, a.re.f, a.re.l);
    a.im.l = fx_fma(s0, a.im.f, a.im.l);
  }
  return true;
}

}  // namespace su3dev
