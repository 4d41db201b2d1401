// su3_fx_kp.cuh -- the SU(2) step of the FP64 update in the arithmetic of
// su3_fx.cuh: the direction of the projected staple, the Kennedy-Pendleton
// proposal and the rotation it makes.
//
// In FP64 instructions these scalars (two logarithms, a cosine, a sine and
// cosine, three square roots and their products: about 150 per subgroup) were
// two thirds of the update's time after its matrix products had left the FP64
// pipe.  The uniforms are integers to begin with, so the logarithm and the
// trigonometric functions take their arguments apart exactly in integers,
// look up 1/2048 of an octave or 1/4096 of a turn, and need three terms of a
// series on what is left, of which only the first two exceed FP32.  Square
// roots start from the hardware's FP32 reciprocal root and take one step of
// third order.  Errors are absolute; the largest measured against long double over
// 200,000 draws, in units of 2^-53 of numbers up to 1: logarithm 1.13 (of up to 37),
// cosine and sine 1.49, root 1.23; root mean squares here / in FP64: direction
// 0.27 / 0.37, a0 0.27 / 0.42, a1 to a3 0.24 / 1.33.
//
// 64-bit integers named x62 hold x in units of 2^-62.
#pragma once

#include "su3_fx.cuh"
#include "su3_fx_tables.cuh"

namespace su3dev {

static __device__ const long long kFxLog[1025] = {SU3_FX_LOG_TABLE};
static __device__ const longlong2 kFxTrig[513] = {SU3_FX_TRIG_TABLE_PAIRS};

#ifndef __CUDA_ARCH__
static const long long kFxLogHost[1025] = {SU3_FX_LOG_TABLE};
static const longlong2 kFxTrigHost[513] = {SU3_FX_TRIG_TABLE_PAIRS};
#endif

SU3_HD long long fx_log_entry(int i) {
#ifdef __CUDA_ARCH__
  return __ldg(&kFxLog[i]);
#else
  return kFxLogHost[i];
#endif
}
SU3_HD longlong2 fx_trig_entry(int i) {
#ifdef __CUDA_ARCH__
  return __ldg(&kFxTrig[i]);
#else
  return kFxTrigHost[i];
#endif
}

// Hardware approximations (about 2^-23); the host's are exact to rounding.
SU3_HD float fx_rcp_approx(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
SU3_HD float fx_rsqrt_approx(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / std::sqrt(x);
#endif
}
SU3_HD int fx_f2i(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)lrintf(x);
#endif
}
SU3_HD int fx_clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// The value of a merged accumulator (unit 2^-60) in units of 2^-62 is 4 times
// it; of an fx, this:
SU3_HD long long fx_to_i62(const fx& a) {
  return (long long)a.h * (1LL << 32) + 2LL * fx_f2i(fx_mul(a.l, 0.5f));
}
// a b for |a b| < 2
SU3_HD fx fx_mulv(const fx& a, const fx& b) {
  facc s = fx_zero();
  fx_mac(s, a, b);
  return fx_norm(s);
}

// The uniform of u01_f64 as the odd integer m, u = m 2^-53.
SU3_HD unsigned long long fx_uniform(uint32_t a, uint32_t b) {
  return (((unsigned long long)a << 21) | (unsigned long long)((b >> 12) << 1)) | 1ull;
}

// -ln(m 2^-53), m odd in [1, 2^53), in units of 2^-57: m 2^-53 = f 2^-E with f in
// [1, 2); C the integer next to 2048 / f, so that f C / 2048 = 1 + r exactly
// with |r| < 2^-10.9, and -ln u = E ln 2 + ln(C / 2048) - ln(1 + r).
SU3_HD long long fx_neg_log(unsigned long long m) {
  const int n = fx_clz64(m);  // 11..63
  const unsigned long long f = m << (n - 11);  // [2^52, 2^53)
  union {
    uint32_t u;
    float f;
  } top, c;
  top.u = 0x3F800000u | ((uint32_t)(f >> 29) & 0x7FFFFFu);
  c.f = fx_fma(fx_rcp_approx(top.f), 2048.0f, 12582912.0f);  // 1.5 2^23: the nearest integer in the low bits
  const uint32_t C = c.u - 0x4B400000u;
  const long long r = (long long)(f * C - (1ull << 63));  // units of 2^-63, |r| < 2^52.2
  const int rh = (int)(r >> 23);                          // units of 2^-40
  const float rf = fx_mul(fx_i2f(rh), 0x1p-40f);
  const float rl = fx_i2f((int)((uint32_t)r & 0x7FFFFFu));  // units of 2^-63
  // r^3/3 - r^4/4 + r^5/5 - rh rl, in units of 2^-57
  const float q = fx_fma(rf, fx_fma(rf, 0.2f, -0.25f), 0x1.555556p-2f);
  const float tail = fx_fma(fx_mul(fx_mul(rf, rf), fx_mul(rf, 0x1p57f)), q, fx_mul(fx_mul(rf, rl), -0x1p-6f));
  const long long log1p = (r >> 6) - (((long long)rh * rh) >> 24) + fx_f2i(tail);
  // E ln 2, ln 2 in units of 2^-57
  return (long long)((unsigned long long)(n - 10) * 0x0162E42FEFA39EF3ull) + fx_log_entry((int)C - 1024) - log1p;
}

// cos and sin of 2 pi m 2^-53 (m < 2^53).
struct fx_cs {
  fx c, s;
};
SU3_HD fx_cs fx_cossin(unsigned long long m) {
  const uint32_t o = (uint32_t)(m >> 50);  // octant; odd ones are mirrored
  unsigned long long w = m & ((1ull << 50) - 1);
  if (o & 1) w = (1ull << 50) - w;
  const int j = (int)((w + (1ull << 40)) >> 41);           // nearest 4096th of a turn, 0..512
  const long long d = (long long)w - ((long long)j << 41);  // |d| <= 2^40, the rest in units of 2^-53 turns
  // t = 2 pi d 2^-53 in units of 2^-62: d 2 pi 2^9, d = dh 2^10 + dl; 2 pi 2^28 = 1686629713.06...
  const int dh = (int)(d >> 10);
  const float dl = fx_i2f((int)((uint32_t)d & 1023u));
  const long long t62 = (((long long)dh * 1686629713LL) >> 9) +
                        fx_f2i(fx_fma(dl, 3216.9908773f, fx_mul(fx_i2f(dh), 1.2744604e-4f)));
  const int th = (int)(t62 >> 21);  // units of 2^-41
  const float tf = fx_mul(fx_i2f(th), 0x1p-41f);
  const float tl = fx_i2f((int)((uint32_t)t62 & 0x1FFFFFu));
  const float t2 = fx_mul(tf, tf);
  // t^2/2 - t^4/24 and t - t^3/6 + t^5/120 (the latter in units of 2^-62: t^3 2^62 / 6)
  const long long v62 = (((long long)th * th) >> 21) + fx_f2i(fx_fma(fx_mul(t2, t2), -0x1p62f / 24.0f, fx_mul(tf, tl)));
  const long long s62 =
      t62 - fx_f2i(fx_mul(fx_mul(fx_mul(tf, 0x1p62f), t2), fx_fma(t2, -1.0f / 120.0f, 1.0f / 6.0f)));
  const longlong2 e = fx_trig_entry(j);
  const fx c0 = fx_from_i62(e.x), s0 = fx_from_i62(e.y), ct = fx_from_i62((1LL << 62) - v62), st = fx_from_i62(s62);
  facc a = fx_zero();
  fx_mac(a, c0, ct);
  fx_msub(a, s0, st);
  facc b = fx_zero();
  fx_mac(b, s0, ct);
  fx_mac(b, c0, st);
  const bool swap = (o + 1) & 2, negc = (o + 2) & 4, negs = o & 4;
  const fx x = fx_norm(a), y = fx_norm(b);
  fx_cs r{swap ? y : x, swap ? x : y};
  r.c = negc ? fx_neg(r.c) : r.c;
  r.s = negs ? fx_neg(r.s) : r.s;
  return r;
}

// (1 - E)^(-1/2) - 1 = E/2 + 3 E^2/8 for E = a merged sum of unit 2^-60, |E| < 2^-20.
SU3_HD fx fx_root_series(long long e60) {
  const float e = fx_mul(fx_i2f((int)(e60 >> 12)), 0x1p-48f);
  return fx_from_i62(2 * e60 + fx_f2i(fx_mul(fx_mul(e, e), 0x1.8p60f)));
}

// 2 sqrt(p (1 - p)) for p62 in [0, 2^62].  The smaller factor is scaled by an even
// power of two into [1/4, 1), so that roots of small numbers are as exact as
// others: q = its product with the larger one in [1/8, 1).  With y the
// approximate reciprocal root of q, w = q y / 2 and E = 1 - q y^2 = 1 - 4 w (y/2):
// sqrt(q) = 2 w (1 - E)^(-1/2).
SU3_HD fx fx_two_root(long long p62) {
  const long long p1 = (1LL << 62) - p62;
  const long long least = p62 < p1 ? p62 : p1;
  if (least <= 0) return fx_make(0, 0.0f);
  const int n = (fx_clz64((unsigned long long)least) - 2) & ~1;  // least << n in [2^60, 2^62)
  const fx q = fx_mulv(fx_from_i62(least << n), fx_from_i62(p62 < p1 ? p1 : p62));
  const float g2 = fx_rsqrt_approx(fx_mul(q.f, 0x1p-30f));  // (1, 2.83]
  const fx g = fx_make(fx_f2i(fx_mul(g2, 0x1p29f)), 0.0f);  // half of it, exactly
  const fx w = fx_mulv(q, g);                               // (0.17, 1/2]
  facc e{1LL << 58, 0.0f};
  fx_msub(e, w, g);                                         // E / 4
  const fx z = fx_root_series(4 * fx_merge(e));
  facc s{0, 0.0f};
  fx_mac(s, w, z);
  const long long r62 = fx_to_i62(w) + 4 * fx_merge(s);  // sqrt(q) / 2
  // 2 sqrt(q 2^-n) = 4 (sqrt(q) / 2) 2^(-n/2); for n = 0 q is at most 1/4
  return fx_from_i62(n ? (2 * r62) >> (n / 2 - 1) : 4 * r62);
}

// Direction and length of the projection 2r (four merged sums rI, 2r = rI 2^-58):
// v = r / |r|, ik = 1 / |2r|; false if it is zero.
SU3_HD bool fx_direction(const long long rI[4], fx v[4], double* ik) {
  unsigned long long any = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) any |= (unsigned long long)(rI[c] ^ (rI[c] >> 63));
  if ((rI[0] | rI[1] | rI[2] | rI[3]) == 0) return false;
  int n = fx_clz64(any | 1ull) - 3;  // the largest |r| into [2^60, 2^61): below 1/2
  long long r[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) r[c] = n >= 0 ? rI[c] << n : rI[c] >> -n;
  fx x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = fx_from_i62(r[c]);
  facc a{0, 0.0f};
#pragma unroll
  for (int c = 0; c < 4; ++c) fx_mac(a, x[c], x[c]);
  long long k60 = fx_merge(a);  // [1/16, 1)
  // |x| doubled where it is below 1/2, and twice where it is next to 1/4 (a power of
  // two along one axis): 1/|x| stays below 2, the end of a real of unit 2^-30
  if (k60 < (1LL << 58) + (1LL << 48)) {
    const int e = k60 < (1LL << 56) + (1LL << 36) ? 2 : 1;
    k60 <<= 2 * e;
    n += e;
    const float f = e == 2 ? 4.0f : 2.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = fx{x[c].h * (1 << e), f * x[c].l, f * x[c].f};
  }
  const fx k = fx_from_i62(4 * k60);  // (1/4 + 2^-22, 1 + 2^-9)
  const float g2 = fx_rsqrt_approx(fx_mul(k.f, 0x1p-30f));
  const fx g = fx_make(fx_f2i(fx_mul(g2, 0x1p29f)), 0.0f);
  const fx w = fx_mulv(k, g);
  facc e{1LL << 58, 0.0f};
  fx_msub(e, w, g);
  const fx z = fx_root_series(4 * fx_merge(e));
  facc s{0, 0.0f};
  fx_mac(s, g, z);
  const long long y62 = 2 * (((long long)g.h << 32) + 4 * fx_merge(s));  // 1/|x|, (0.998, 2 - 2^-21)
  const fx y = fx_from_i62(y62);
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = fx_mulv(x[c], y);
  // |2r| = |x| 2^(4 - n)
#ifdef __CUDA_ARCH__
  const double yd = __ll2double_rn(y62);
  *ik = __hiloint2double(__double2hiint(yd) + (n - 4 - 62) * (1 << 20), __double2loint(yd));
#else
  *ik = std::ldexp((double)y62, n - 4 - 62);
#endif
  return true;
}

// A Kennedy-Pendleton proposal from the uniforms m[0..5] (odd integers, u = m
// 2^-53): delta = -(ln u0 + cos^2(2 pi u1) ln u2) / alpha; accepted if u3^2 <= 1 -
// delta/2, then a0 = 1 - delta and a1..a3 on the sphere of radius sqrt(1 -
// a0^2) in the direction of u4, u5.  fx_draw is the part that does not depend
// on the staple, fx_propose the rest.
struct fx_drawn {
  long long S;   // -ln u0 - cos^2 ln u2 in units of 2^-56
  long long u3;  // u3 in units of 2^-62
  fx d[3];       // direction: sin(theta) cos(phi), sin(theta) sin(phi), cos(theta)
};
SU3_HD fx_drawn fx_draw(const unsigned long long m[6]) {
  fx_drawn r;
  // cos^2 = (1 + cos(4 pi u1)) / 2; the two logarithms and the two angles in one
  // piece of code (instruction cache)
  long long l0 = 0, l2 = 0;
  fx_cs c2{}, phi{};
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
  for (int n = 0; n < 2; ++n) {
    l0 = l2;
    c2 = phi;
    l2 = fx_neg_log(n == 0 ? m[0] : m[2]);
    phi = fx_cossin(n == 0 ? (m[1] << 1) & ((1ull << 53) - 1) : m[5]);
  }
  const fx cc = fx_from_i62((fx_to_i62(c2.c) + (1LL << 62)) >> 1);
  // S is at most 74; cos^2's integer part times both words of the second logarithm
  // (up to 37: its low word is too large for an FP32 part)
  const int l2l = (int)(uint32_t)l2, l2h = (int)(l2 >> 32) + (int)((uint32_t)l2l >> 31);
  r.S = (l0 >> 1) + (((long long)cc.h * l2h) << 1) + (((long long)cc.h * l2l) >> 31) +
        fx_f2i(fx_mul(fx_mul(cc.l, 0x1p-31f), fx_i2f(l2h)));
  r.u3 = (long long)(m[3] << 9);
  const long long u4 = (long long)(m[4] << 9);
  const fx sn = fx_two_root(u4);
  r.d[0] = fx_mulv(sn, phi.c);
  r.d[1] = fx_mulv(sn, phi.s);
  r.d[2] = fx_from_i62((1LL << 62) - 2 * u4);
  return r;
}
SU3_HD bool fx_propose(const fx_drawn& w, double inv_alpha, fx a[4]) {
#ifdef __CUDA_ARCH__
  const double Sd = __ll2double_rn(w.S);
#else
  const double Sd = (double)w.S;
#endif
  const double delta = Sd * 0x1p-56 * inv_alpha;
  if (!(delta < 2.0)) return false;
  const long long p62 = fx_i62_from_double(delta) >> 1;  // delta / 2
  const fx u3 = fx_from_i62(w.u3);
  facc t{0, 0.0f};
  fx_mac(t, u3, u3);
  if (fx_merge(t) > (1LL << 60) - (p62 >> 2)) return false;
  const fx rho = fx_two_root(p62);
  a[0] = fx_from_i62((1LL << 62) - 2 * p62);
#pragma unroll
  for (int c = 0; c < 3; ++c) a[c + 1] = fx_mulv(rho, w.d[c]);
  return true;
}

// R = Y V^+, Y = m(a), V = m(v), m(q) = [[q0 + i q3, q2 + i q1], [-q2 + i q1, q0 - i q3]]:
// its first row (R00, R01); R10 = -conj(R01), R11 = conj(R00).
SU3_HD void fx_rotation(const fx a[4], const fx v[4], cfx& R00, cfx& R01) {
  facc s = fx_zero();
  fx_mac(s, a[0], v[0]);
  fx_mac(s, a[1], v[1]);
  fx_mac(s, a[2], v[2]);
  fx_mac(s, a[3], v[3]);
  R00.re = fx_norm(s);
  s = fx_zero();
  fx_mac(s, a[3], v[0]);
  fx_msub(s, a[0], v[3]);
  fx_mac(s, a[1], v[2]);
  fx_msub(s, a[2], v[1]);
  R00.im = fx_norm(s);
  s = fx_zero();
  fx_msub(s, a[0], v[2]);
  fx_mac(s, a[3], v[1]);
  fx_mac(s, a[2], v[0]);
  fx_msub(s, a[1], v[3]);
  R01.re = fx_norm(s);
  s = fx_zero();
  fx_msub(s, a[3], v[2]);
  fx_msub(s, a[0], v[1]);
  fx_mac(s, a[1], v[0]);
  fx_mac(s, a[2], v[3]);
  R01.im = fx_norm(s);
}

}  // namespace su3dev
