// su3_update.cuh -- one checkerboard link update on sm_103a CUDA cores, shared
// by the single-lattice half-sweep kernels (one launch per (mu, parity)) and
// the persistent batched sweep.
//
// A link U_mu(x) gathers its six-staple sum from the 18 neighbouring links,
// runs the one-hit Kennedy-Pendleton heatbath in the SU(2) subgroups (0,1),
// (0,2), (1,2) (Cabibbo-Marinari), is reunitarised and stored.  Links of one
// (mu, parity) never enter each other's staples (checkerboard updating,
// Abstract and Sec. 1 of Berg & Wu, arXiv:0904.1179); every update draws its
// random numbers from Philox counters keyed by its site, so the result does
// not depend on which thread, block or launch performs it.  The work is a 4D
// stencil of 3x3 complex products, not a dense contraction: CUDA cores, no
// tensor cores.
#pragma once

#include "su3_device.cuh"
#include "su3_fx.cuh"
#include "su3_fx_kp.cuh"
#include "su3_pair.cuh"

namespace su3dev {

constexpr double kTwoPi = 6.283185307179586476925286766559;

template <typename T>
__device__ __forceinline__ mat3<T> zero3() {
  mat3<T> m;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) m.e[i][k] = mk(T(0), T(0));
  return m;
}

// The FP32 stores come in two layouts: one site per float4 column group (the
// single-site layout) and the site-paired layout of su3_sitepair.cuh, which
// stores the sites x and x + (L3/2) e3 of a lattice whose L3 is a multiple of
// 4 side by side.  Single-site code reads and writes the latter one site at a
// time (PAIRS = true); Vh is the full lattice's half volume in both.
template <bool CG, bool PAIRS>
__device__ __forceinline__ pm3 load_pm3_l(const float4* __restrict__ U, int mu, int p, int h, int Vh) {
  if constexpr (PAIRS) {
    const int Vp = Vh / 2;
    const int half = h >= Vp ? 1 : 0;
    pm3 m;
    if (!link_ok(mu, p, h, Vh)) {
#pragma unroll
      for (int k = 0; k < 3; ++k) m.re[k] = m.im[k] = make_float2(0.f, 0.f);
      return m;
    }
    const float* b = (const float*)(U + pair_offset(mu, p, h - half * Vp, Vp)) + half;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float* e0 = b + 4 * kPairTile * k;        // entry (row 0, column k)
      const float* e1 = b + 4 * kPairTile * (3 + k);  // entry (row 1, column k)
      m.re[k] = make_float2(CG ? __ldcg(e0) : __ldg(e0), CG ? __ldcg(e1) : __ldg(e1));
      m.im[k] = make_float2(CG ? __ldcg(e0 + 2) : __ldg(e0 + 2), CG ? __ldcg(e1 + 2) : __ldg(e1 + 2));
    }
    return m;
  } else {
    return load_pm3<CG>(U, mu, p, h, Vh);
  }
}

// Single-site access to a site-paired store: rows 0,1 of site h's link (mu, p)
// as 12 floats, row 0 then row 1, (re, im) per column (as store_f32_rows01
// takes them); Vp = V/4 pairs per (mu, parity), pair h mod Vp, member h / Vp.
__device__ __forceinline__ void load_pair_site(const float4* __restrict__ U, int mu, int p, int h, int Vp, float r[12]) {
  if (!link_ok(mu, p, h, 2LL * Vp)) {
#pragma unroll
    for (int c = 0; c < 12; ++c) r[c] = 0.f;
    return;
  }
  const int half = h >= Vp ? 1 : 0;
  const float* b = (const float*)(U + pair_offset(mu, p, h - half * Vp, Vp)) + half;
#pragma unroll
  for (int e = 0; e < 6; ++e) {
    r[6 * (e / 3) + 2 * (e % 3)] = __ldg(b + 4 * kPairTile * e);
    r[6 * (e / 3) + 2 * (e % 3) + 1] = __ldg(b + 4 * kPairTile * e + 2);
  }
}

__device__ __forceinline__ void store_pair_site(float4* U, int mu, int p, int h, int Vp, const float r[12]) {
  if (!link_ok(mu, p, h, 2LL * Vp)) return;
  const int half = h >= Vp ? 1 : 0;
  float* b = (float*)(U + pair_offset(mu, p, h - half * Vp, Vp)) + half;
#pragma unroll
  for (int e = 0; e < 6; ++e) {
    b[4 * kPairTile * e] = r[6 * (e / 3) + 2 * (e % 3)];
    b[4 * kPairTile * e + 2] = r[6 * (e / 3) + 2 * (e % 3) + 1];
  }
}

// Six-staple sum A for U_mu(x), x = st of parity p:
//   sum_{nu != mu} U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+ + U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu).
// Each three-link path is an SU(3) matrix, so only its rows 0 and 1 are
// multiplied out; its row 2, conj(row0 x row1), is formed inside the
// accumulation of A's row 2 (acc_completed).  The paths are added in the
// order forward, backward for nu ascending; every floating-point kernel that
// forms a staple keeps this order, so their results agree bit for bit.
// The two three-link paths of direction nu (nu != mu), rows 0,1, in FP64
// arithmetic (update_link_f64_far; links through L2, as other blocks of the
// same launch may have written them):
//   forward  F = U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+,
//   backward B = U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu).
// h_pmu is the half index of x + mu-hat.
template <typename G>
__device__ __forceinline__ mat3<double> forward_path(const G& g, const double2* U, int h, int p, int mu, int nu, int h_pmu,
                                                     int h_pnu) {
  const int q = p ^ 1;
  const mat3<double> a = load_f64<true>(U, nu, q, h_pmu, g.Vh);  // U_nu(x+mu)
  const mat3<double> b = load_f64<true>(U, mu, q, h_pnu, g.Vh);  // U_mu(x+nu)
  mat3<double> t;
  mul_nd_rows01(a, b, t);
  const mat3<double> c = load_f64<true>(U, nu, p, h, g.Vh);  // U_nu(x)
  mat3<double> f;
  mul_nd_rows01(t, c, f);
  return f;
}

template <typename G>
__device__ __forceinline__ mat3<double> backward_path(const G& g, const double2* U, int p, int mu, int nu, int h_mnu,
                                                      int h_pmu_mnu) {
  const int q = p ^ 1;
  const mat3<double> d = load_f64<true>(U, nu, p, h_pmu_mnu, g.Vh);  // U_nu(x+mu-nu)
  const mat3<double> e = load_f64<true>(U, mu, q, h_mnu, g.Vh);      // U_mu(x-nu)
  // Rows 0,1 of d^+ e^+ = (e d)^+ are the conjugated columns 0,1 of e d, which
  // need all three rows of e (stored in full here) but no row-2 completion.
  mat3<double> hm;
  mul_nn_cols01(e, d, hm);
  const mat3<double> f = load_f64<true>(U, nu, q, h_mnu, g.Vh);  // U_nu(x-nu)
  mat3<double> b;
  mul_dn_rows01(hm, f, b);
  return b;
}

// 2x2 block of W = U A in rows/columns (i, j), projected on the SU(2) direction,
// returned as 2r = (Re(W_ii+W_jj), Im(W_ij+W_ji), Re(W_ij-W_ji), Im(W_ii-W_jj)):
// the factor 1/2 of r cancels in r/|r| and is folded into 1/alpha.
template <typename T>
__device__ __forceinline__ void su2_projection(const mat3<T>& u, const mat3<T>& A, int i, int j, T r[4]) {
  cx<T> wii = mk(T(0), T(0)), wij = wii, wji = wii, wjj = wii;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    wii = mac(wii, u.e[i][c], A.e[c][i]);
    wij = mac(wij, u.e[i][c], A.e[c][j]);
    wji = mac(wji, u.e[j][c], A.e[c][i]);
    wjj = mac(wjj, u.e[j][c], A.e[c][j]);
  }
  r[0] = wii.re + wjj.re;
  r[1] = wij.im + wji.im;
  r[2] = wij.re - wji.re;
  r[3] = wii.im - wjj.im;
}

// rows (i, j) of u <- R rows (i, j), R = Y V^+ with Y = m(a), V = m(v),
// m(q) = [[q0 + i q3, q2 + i q1], [-q2 + i q1, q0 - i q3]].
// rows_j = false leaves row j unchanged (its new value is not needed).
template <typename T>
__device__ __forceinline__ void apply_su2(mat3<T>& u, int i, int j, const T a[4], const T v[4], bool rows_j = true) {
  const cx<T> y00 = mk(a[0], a[3]), y01 = mk(a[2], a[1]);
  const cx<T> v00 = mk(v[0], v[3]), v01 = mk(v[2], v[1]), v10 = mk(-v[2], v[1]), v11 = mk(v[0], -v[3]);
  // (V^+)_{pq} = conj(V_{qp}); a product of two matrices of this SU(2) form
  // has the form again, so R10 = -conj(R01) and R11 = conj(R00).
  const cx<T> R00 = mac_cb(mac_cb(mk(T(0), T(0)), y00, v00), y01, v01);
  const cx<T> R01 = mac_cb(mac_cb(mk(T(0), T(0)), y00, v10), y01, v11);
  const cx<T> R10 = mk(-R01.re, R01.im);
  const cx<T> R11 = mk(R00.re, -R00.im);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cx<T> ui = u.e[i][c], uj = u.e[j][c];
    u.e[i][c] = mac(mul(R00, ui), R01, uj);
    if (rows_j) u.e[j][c] = mac(mul(R10, ui), R11, uj);
  }
}

__device__ __forceinline__ int subrow_i(int sub) { return sub == 2 ? 1 : 0; }
__device__ __forceinline__ int subrow_j(int sub) { return sub == 0 ? 1 : 2; }


// Parameters of one link update that do not vary across the links of a lattice.
struct UpdateConsts {
  double three_over_beta_f64;  // 3 / beta: 1/alpha = 3 / (2 beta k) = three_over_beta / (2k)
  float three_over_beta;
  int max_tries;  // 1: one-hit heatbath; > 1: repeat until accepted, at most this many proposals
  int* far;       // FP64 stores: the flags of SweepState (su3_device.cuh)
};

// Accepted and drawn SU(2) proposals of one link update (a degenerate
// subgroup counts as one proposal).
struct UpdateCount {
  int accepted, proposed;
};

// Kennedy-Pendleton proposals of subgroup sub of link (s, mu) at sweep t in
// FP64: a0..a3 of the accepted one into a; false if none of the ntries was.
template <bool REPEAT, typename KEY>
__device__ __forceinline__ bool propose_f64(uint32_t s, int mu, int sub, uint64_t t, const KEY& key, double inv_alpha,
                                            int max_tries, double a[4], UpdateCount& cnt) {
  const int ntries = REPEAT ? max_tries : 1;
  for (int tr = 0; tr < ntries; ++tr) {
    double uu[6];
#pragma unroll
    for (int call = 0; call < 3; ++call) {
      const uint32_t w1 = (uint32_t)(mu | (sub << 2) | (call << 4)) | ((uint32_t)tr << 6);
      const uint4 w = philox4x32_10(rng_counter(s, w1, t, kTagUpdate), key);
      uu[2 * call] = u01_f64(w.x, w.y);
      uu[2 * call + 1] = u01_f64(w.z, w.w);
    }
    ++cnt.proposed;
    const double c = cospi(2.0 * uu[1]);  // cos(2 pi u1)
    const double delta = -(log_u01(uu[0]) + c * c * log_u01(uu[2])) * inv_alpha;
    if (uu[3] * uu[3] > 1.0 - 0.5 * delta) continue;
    const double a0 = 1.0 - delta;
    double rho = 1.0 - a0 * a0;
    rho = rho > 0.0 ? sqrt(rho) : 0.0;
    const double ct = 1.0 - 2.0 * uu[4];
    double sn = 1.0 - ct * ct;
    sn = sn > 0.0 ? sqrt(sn) : 0.0;
    double sphi, cphi;
    sincospi(2.0 * uu[5], &sphi, &cphi);  // angle 2 pi u5
    a[0] = a0;
    a[1] = rho * sn * cphi;
    a[2] = rho * sn * sphi;
    a[3] = rho * ct;
    ++cnt.accepted;
    return true;
  }
  return false;
}

// ---------------------------------------------------------------------------
// One FP64 link update in FP64 arithmetic: staple, three SU(2) heatbath steps,
// Gram-Schmidt, store.  It serves configurations with links far from SU(3)
// (SweepState::far), whose entries and products may leave the range of
// su3_fx.cuh: one function for every direction and heatbath, not inlined and
// its loops not unrolled, since no sweep of a proper configuration runs it.
// Links are read through L2: blocks of the same launch may have written them.
// meas (nullptr: off) receives (1/3) Re Tr(U_new A_<), A_< the staple terms of
// the directions nu < mu.
// G: Geometry (periodic lattice) or SubGeometry (sublattice with ghost
// layers); h enumerates the sites of parity p.
// ---------------------------------------------------------------------------
template <typename KEY, typename G>
__device__ __noinline__ UpdateCount update_link_f64_far(const G& g, double2* U, int h, int p, int mu, uint64_t t,
                                                        const KEY& key, const UpdateConsts& uc, double* meas) {
  const auto st = site_of(g, h, p);
  const uint32_t s = (uint32_t)canon(g, st);
  h = store_index(g, st, h);
  mat3<double> A = zero3<double>(), Apart = A;
  const int h_pmu = nb_half_rt(g, st, mu, +1);
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    acc_completed(A, forward_path(g, U, h, p, mu, nu, h_pmu, nb_half_rt(g, st, nu, +1)));
    acc_completed(A, backward_path(g, U, p, mu, nu, nb_half_rt(g, st, nu, -1), nb_half2_rt(g, st, mu, nu)));
    if (nu == mu - 1) Apart = A;
  }
  UpdateCount cnt{0, 0};
  mat3<double> u = load_f64<true>(U, mu, p, h, g.Vh);
#pragma unroll 1
  for (int sub = 0; sub < 3; ++sub) {
    const int i = subrow_i(sub), j = subrow_j(sub);
    double r[4];  // 2r
    su2_projection(u, A, i, j, r);
    const double kk = r[0] * r[0] + r[1] * r[1] + r[2] * r[2] + r[3] * r[3];  // (2k)^2
    if (!(kk > 0.0)) {  // k = 0: degenerate staple (measure zero), leave the subgroup
      ++cnt.proposed;
      continue;
    }
    const double ik = rsqrt(kk);                           // 1 / (2k)
    const double inv_alpha = uc.three_over_beta_f64 * ik;  // 1/alpha = 3 / (2 beta k)
    double a[4];
    if (!propose_f64<true>(s, mu, sub, t, key, inv_alpha, uc.max_tries, a, cnt)) continue;
    const double v[4] = {r[0] * ik, r[1] * ik, r[2] * ik, r[3] * ik};  // r / k
    // Row 2 leaves the last subgroup unused: reunitarisation rebuilds it.
    apply_su2(u, i, j, a, v, sub < 2);
  }
  cx<double> r0[3] = {u.e[0][0], u.e[0][1], u.e[0][2]};
  cx<double> r1[3] = {u.e[1][0], u.e[1][1], u.e[1][2]};
  gram_schmidt_rows01(r0, r1);
  mat3<double> out;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    out.e[0][k] = r0[k];
    out.e[1][k] = r1[k];
  }
  complete_row2(out);
  store_f64(U, mu, p, h, g.Vh, out);
  if (far_from_su3(out)) atomicOr(uc.far + 1, 1);
  if (meas) {
    double tr = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) tr = fma(out.e[i][k].re, Apart.e[k][i].re, fma(-out.e[i][k].im, Apart.e[k][i].im, tr));
    *meas = tr * (1.0 / 3.0);
  }
  return cnt;
}

// ---------------------------------------------------------------------------
// cp.async: 16-byte copies from global to shared memory that do not pass
// through registers, tracked in commit groups per thread.
// ---------------------------------------------------------------------------
// Both forms copy through L1 (.ca): cache operators are performance hints
// and do not change the memory-consistency behaviour, so links written by
// other blocks of a persistent launch are seen once the block has acquired
// their completion counts; and on GB300 the L1-bypassing cp.async.cg made the
// site-paired sweep 1.7 times slower.
template <bool CG>
__device__ __forceinline__ void cp_async16(uint32_t saddr, const float4* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(saddr), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async16(double2* dst, const double2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// The FP64 link update on the integer and FP32 pipes (su3_fx.cuh): links are
// read from the FP64 store, split into integer and FP32 parts, and multiplied
// there; the SU(2) steps (su3_fx_kp.cuh) use it too, but for the four FP64
// operations that make delta from 1/alpha, whose range beta leaves open.
// ---------------------------------------------------------------------------
// Two rows' entries side by side: their FP32 parts go through the paired FMA
// (one instruction for both), each half rounded like fx_mac's.
struct fx2 {
  int h[2];
  float2 l, f;
};
struct cfx2 {
  fx2 re, im;
};
struct facc2 {
  long long hh[2];
  float2 c;
};
struct cfacc2 {
  facc2 re, im;
};
__device__ __forceinline__ fx2 fx2_of(const fx& a, const fx& b) {
  return fx2{{a.h, b.h}, make_float2(a.l, b.l), make_float2(a.f, b.f)};
}
__device__ __forceinline__ cfx2 cfx2_of(const cfx& a, const cfx& b) { return cfx2{fx2_of(a.re, b.re), fx2_of(a.im, b.im)}; }
__device__ __forceinline__ fx fx2_row(const fx2& a, int i) {
  return i ? fx{a.h[1], a.l.y, a.f.y} : fx{a.h[0], a.l.x, a.f.x};
}
__device__ __forceinline__ cfx cfx2_row(const cfx2& a, int i) { return cfx{fx2_row(a.re, i), fx2_row(a.im, i)}; }
__device__ __forceinline__ void fx2_set(fx2& a, int i, const fx& b) {
  a.h[i] = b.h;
  (i ? a.l.y : a.l.x) = b.l;
  (i ? a.f.y : a.f.x) = b.f;
}
__device__ __forceinline__ void cfx2_set(cfx2& a, int i, const fx& re, const fx& im) {
  fx2_set(a.re, i, re);
  fx2_set(a.im, i, im);
}
__device__ __forceinline__ cfacc2 cfx2_zero() {
  const facc2 z{{1LL << 29, 1LL << 29}, make_float2(0.0f, 0.0f)};
  return cfacc2{z, z};
}
__device__ __forceinline__ void fx2_mac(facc2& s, const fx2& a, const fx& b) {
  s.hh[0] += (long long)a.h[0] * b.h;
  s.hh[1] += (long long)a.h[1] * b.h;
  s.c = fma2(a.f, bc2(b.l), s.c);
  s.c = fma2(a.l, bc2(b.f), s.c);
}
__device__ __forceinline__ void fx2_msub(facc2& s, const fx2& a, const fx& b) {
  const int n = -b.h;
  s.hh[0] += (long long)a.h[0] * n;
  s.hh[1] += (long long)a.h[1] * n;
  s.c = fma2(a.f, bc2(-b.l), s.c);
  s.c = fma2(a.l, bc2(-b.f), s.c);
}
__device__ __forceinline__ void cfx2_mac(cfacc2& s, const cfx2& a, const cfx& b) {
  fx2_mac(s.re, a.re, b.re);
  fx2_msub(s.re, a.im, b.im);
  fx2_mac(s.im, a.re, b.im);
  fx2_mac(s.im, a.im, b.re);
}

// A link entry of the store, split.  Real parts on the integer pipe (14
// instructions), imaginary parts by a conversion on the FP64 pipe (5, but 16 SM
// cycles of a pipe that is otherwise nearly idle): 32^4 3.20 ms per sweep, against
// 3.74 with both converted (and, on an earlier kernel, 3.90 against 4.17 with
// both on the integer pipe).
__device__ __forceinline__ cfx fx_entry(double2 v, uint32_t flip) {
  return cfx{fx_from_double(v.x), fx_from_double_cvt(v.y, flip)};
}

// A link of the store, or its adjoint, entry by entry.
struct FxLink {
  const double2* b;
  uint32_t si, sk;  // elements between rows and between columns
  // (an access that the bounds-checked build finds out of range reads link 0)
  __device__ __forceinline__ FxLink(const void* U, int mu, int p, int h, int Vh, bool dag = false)
      : b((const double2*)U + link_base(mu, p, Vh, kEntriesF64) + (link_ok(mu, p, h, Vh) ? h : 0)),
        si(dag ? (uint32_t)Vh : 3u * (uint32_t)Vh),
        sk(dag ? 3u * (uint32_t)Vh : (uint32_t)Vh) {}
  // 9 Vh < 2^32
  __device__ __forceinline__ const double2* at(int i, int k) const { return b + (size_t)((uint32_t)i * si + (uint32_t)k * sk); }
};

// The links of a path pass through shared memory: each thread owns three slots,
// for rows 0,1 of X and for Y and Z, and requests the next path's link with 16-byte
// cp.async copies once it has read the slot, so that three links are in flight
// behind the arithmetic (the code of a path is rolled up for the instruction
// caches and loads nothing ahead by itself).  Strides of 7 and 9 double2: eight
// lanes' 16-byte reads touch every bank once.  Dynamic shared memory,
// kFxThreadBytes per thread.
// After the slots: the thread's half-index steps along the eight directions
// (FxSteps).
constexpr int kFxSlotBytes = (7 + 9 + 9) * 16;
constexpr int kFxThreadBytes = kFxSlotBytes + 8 * 4;

struct FxRing {
  double2 *x, *yz;  // this thread's slot of X, and of Y; Z is `step` further
  int step;
  __device__ __forceinline__ FxRing() {
    extern __shared__ double2 fx_ring[];
    const int n = blockDim.x, t = threadIdx.x;
    x = fx_ring + 7 * t;
    yz = fx_ring + 7 * n + 9 * t;
    step = 9 * n;
  }
  __device__ __forceinline__ void fetch_rows01(const FxLink& l) const {
#pragma unroll
    for (int e = 0; e < 6; ++e) cp_async16(x + e, l.at(e / 3, e % 3));
  }
  __device__ __forceinline__ void fetch(int slot, const FxLink& l) const {
#pragma unroll
    for (int e = 0; e < 9; ++e) cp_async16(yz + slot * step + e, l.at(e / 3, e % 3));
  }
};

// Changes of a site's half index for a step up and down along each direction:
// half indices are separable, so x + mu - nu adds two of them.  Looked up by
// direction at run time.
struct FxSteps {
  int* d;
  int n;
  __device__ __forceinline__ FxSteps() {
    extern __shared__ double2 fx_ring[];
    n = blockDim.x;
    d = (int*)((char*)fx_ring + (size_t)n * kFxSlotBytes) + threadIdx.x;
  }
  template <typename G, typename S>
  __device__ __forceinline__ void set(const G& g, const S& st, int h) const {
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
      d[nu * n] = nb_half(g, st, nu, +1) - h;
      d[(4 + nu) * n] = nb_half(g, st, nu, -1) - h;
    }
  }
  __device__ __forceinline__ int at(int nu, bool down) const { return d[(nu + (down ? 4 : 0)) * n]; }
};

// The two paths of direction nu (forward_path, backward_path above) have one
// form, X Y^+ Z:
//   forward:  U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+,  backward: U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu),
// number 2 n and 2 n + 1 for the n-th direction nu != mu.  hx, hy, hz: half indices.
struct FxPath {
  int nu, hx, hy, hz;
  bool backward;
  __device__ __forceinline__ FxPath(const FxSteps& steps, int h, int mu, int path) {
    backward = path & 1;
    nu = (path >> 1) + ((path >> 1) >= mu ? 1 : 0);
    const int o = steps.at(nu, backward);
    hy = h + o;
    hx = h + steps.at(mu, false) + (backward ? o : 0);
    hz = backward ? hy : h;
  }
  __device__ __forceinline__ FxLink X(const void* U, int p, int Vh) const {
    return FxLink(U, nu, backward ? p : p ^ 1, hx, Vh, backward);
  }
  __device__ __forceinline__ FxLink Yd(const void* U, int p, int mu, int Vh) const {
    return FxLink(U, mu, p ^ 1, hy, Vh, true);
  }
  __device__ __forceinline__ FxLink Z(const void* U, int p, int Vh) const {
    return FxLink(U, nu, backward ? p ^ 1 : p, hz, Vh, !backward);
  }
};

// Adds the paths first .. last - 1 of U_mu(x), x = st of parity p stored at h, to A;
// own (optional): a link that ends up in the ring's slot of Y (cp_async_wait<0>).
// Apart (optional): receives the sum of the terms with nu < mu.  After the
// update, Re Tr(U_new Apart) is the sum of the plaquettes of the planes
// (mu, nu < mu) at x and at x - nu-hat.
template <typename G, typename S>
__device__ __forceinline__ void staple_paths_fx(fx_staple& A, const G& g, const void* U, const S& st, int h, int p,
                                                int mu, int first, int last, const FxRing& ring, const FxLink* own,
                                                fx_mat* Apart = nullptr) {
  const FxSteps steps;
  steps.set(g, st, h);
  {
    const FxPath t(steps, h, mu, first);
    ring.fetch_rows01(t.X(U, p, g.Vh));
    cp_async_commit();
    ring.fetch(0, t.Yd(U, p, mu, g.Vh));
    cp_async_commit();
    ring.fetch(1, t.Z(U, p, g.Vh));
    cp_async_commit();
  }
// A forward and a backward path per turn: their directions are then known to the
// compiler (GB300, ms per sweep with 1 / 2 / 6 paths per turn: 16^4 0.281 / 0.270 /
// 0.267, 24^4 1.119 / 1.096 / 1.075, 32^4 3.198 / 3.184 / 3.342, where the code no
// longer fits the instruction caches).
#pragma unroll 2
  for (int path = first; path < last; ++path) {
    const bool backward = path & 1, more = path + 1 < last;
    const FxPath t(steps, h, mu, more ? path + 1 : path);
    cfx2 f[3];  // rows 0,1
    cp_async_wait<2>();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t flip = backward ? 0x80000000u : 0u;
      f[k] = cfx2_of(fx_entry(ring.x[k], flip), fx_entry(ring.x[3 + k], flip));
    }
    if (more) ring.fetch_rows01(t.X(U, p, g.Vh));
    cp_async_commit();
    // the two products in one piece of code
#pragma unroll 1
    for (int n = 0; n < 2; ++n) {
      const double2* z = ring.yz + n * ring.step;
      const uint32_t flip = n == 0 || !backward ? 0x80000000u : 0u;
      cfx2 q[3];
      cp_async_wait<2>();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        cfacc2 s = cfx2_zero();
#pragma unroll
        for (int j = 0; j < 3; ++j) cfx2_mac(s, f[j], fx_entry(z[3 * j + k], flip));
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const long long re = fx_merge(facc{s.re.hh[i], i ? s.re.c.y : s.re.c.x}),
                          im = fx_merge(facc{s.im.hh[i], i ? s.im.c.y : s.im.c.x});
          cfx2_set(q[k], i, fx_norm_merged(re), fx_norm_merged(im));
          A.r[i][k][0] += n ? re : 0;  // the path's rows 0,1
          A.r[i][k][1] += n ? im : 0;
        }
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) f[k] = q[k];
      if (more)
        ring.fetch(n, n == 0 ? t.Yd(U, p, mu, g.Vh) : t.Z(U, p, g.Vh));
      else if (own && n == 0)
        ring.fetch(0, *own);
      cp_async_commit();
    }
    fx_rows01 F;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      F.e[0][k] = cfx2_row(f[k], 0);
      F.e[1][k] = cfx2_row(f[k], 1);
    }
    fx_staple_add_row2(A, F);
    if (Apart && backward && (path >> 1) == mu - 1) *Apart = fx_staple_mat(A, path + 1);
  }
}

// A sum of products of units 2^-30 and 2^-28 merged (units of 2^-58).  The cross
// terms of the projection and of the measured trace reach 2^65.4 in units of
// 2^-90: they are taken to 2^-54.
__device__ __forceinline__ long long fx_merge_wide(const facc& s) {
  return s.hh + 16LL * __float2int_rn(__fmul_rn(s.c, 0x1p-36f));
}

// Column c's part of 2r (su2_projection), merged (units of 2^-58): u_ic, u_jc and
// A_ci, A_cj.
__device__ __forceinline__ void fx_projection_column(const cfx& ui, const cfx& uj, const cfx& ai, const cfx& aj,
                                                     long long r[4]) {
  facc w[4] = {{0, 0.0f}, {0, 0.0f}, {0, 0.0f}, {0, 0.0f}};
  fx_mac(w[0], ui.re, ai.re);
  fx_msub(w[0], ui.im, ai.im);
  fx_mac(w[0], uj.re, aj.re);
  fx_msub(w[0], uj.im, aj.im);
  fx_mac(w[1], ui.re, aj.im);
  fx_mac(w[1], ui.im, aj.re);
  fx_mac(w[1], uj.re, ai.im);
  fx_mac(w[1], uj.im, ai.re);
  fx_mac(w[2], ui.re, aj.re);
  fx_msub(w[2], ui.im, aj.im);
  fx_msub(w[2], uj.re, ai.re);
  fx_mac(w[2], uj.im, ai.im);
  fx_mac(w[3], ui.re, ai.im);
  fx_mac(w[3], ui.im, ai.re);
  fx_msub(w[3], uj.re, aj.im);
  fx_msub(w[3], uj.im, aj.re);
#pragma unroll
  for (int n = 0; n < 4; ++n) r[n] = fx_merge_wide(w[n]);
}

// Entries of one column of the two rows that R turns (R10 = -conj(R01), R11 =
// conj(R00)).
__device__ __forceinline__ void fx_rotate_column(const cfx& R00, const cfx& R01, cfx& ui, cfx& uj) {
  const cfx2 Ri = cfx2_of(R00, cfx{fx_neg(R01.re), R01.im}), Rj = cfx2_of(R01, cfx_conj(R00));
  cfacc2 z = cfx2_zero();
  cfx2_mac(z, Ri, ui);
  cfx2_mac(z, Rj, uj);
  ui = cfx{fx_norm(facc{z.re.hh[0], z.re.c.x}), fx_norm(facc{z.im.hh[0], z.im.c.x})};
  uj = cfx{fx_norm(facc{z.re.hh[1], z.re.c.y}), fx_norm(facc{z.im.hh[1], z.im.c.y})};
}

// The uniforms of proposal tr of subgroup sub.
template <typename KEY>
__device__ __forceinline__ fx_drawn fx_draw_at(uint32_t s, int mu, int sub, int tr, uint64_t t, const KEY& key) {
  unsigned long long m[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int call = 0; call < 3; ++call) {
    const uint32_t w1 = (uint32_t)(mu | (sub << 2) | (call << 4)) | ((uint32_t)tr << 6);
    const uint4 b = philox4x32_10(rng_counter(s, w1, t, kTagUpdate), key);
#pragma unroll
    for (int n = 0; n < 4; ++n) m[n] = m[n + 2];
    m[4] = fx_uniform(b.x, b.y);
    m[5] = fx_uniform(b.z, b.w);
  }
  return fx_draw(m);
}

// Everything after the staple A0 (unit 2^-28) of the link u: three SU(2) heatbath steps,
// reunitarisation, the store of link (s, mu) at storage half index h.
// MEAS: also (1/3) Re Tr(U_new Apart) into *meas.
template <bool REPEAT, bool MEAS, typename KEY, typename G>
__device__ __forceinline__ UpdateCount heatbath_fx(const G& g, double2* U, int h, int p, int mu, uint64_t t, uint32_t s,
                                                   const KEY& key, const UpdateConsts& uc, fx_mat u, const fx_mat& A0,
                                                   const fx_mat& Apart, double* meas) {
  UpdateCount cnt{0, 0};
  // The subgroups (0,1), (0,2), (1,2) in one piece of code (instruction cache):
  // the step always acts on rows 0, 1 of u and columns 0, 1 of A, and between the
  // steps rows and columns change places: orders (0,1,2), (0,2,1), (1,2,0).
  // They are kept without f, which the uses convert again: 36 registers.
  cfxs us[3][3], A[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      us[i][k] = cfx_short(u.e[i][k]);
      A[i][k] = cfx_short(A0.e[i][k]);
    }
#pragma unroll 1
  for (int sub = 0; sub < 3; ++sub) {
    long long r[4] = {0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      long long q[4];
      fx_projection_column(cfx_of(us[0][c]), cfx_of(us[1][c]), cfx_of(A[c][0]), cfx_of(A[c][1]), q);
#pragma unroll
      for (int n = 0; n < 4; ++n) r[n] += q[n];
    }
    fx v[4], a[4];
    double ik;
    bool accepted = false;
    if (fx_direction(r, v, &ik)) {
      const double inv_alpha = uc.three_over_beta_f64 * ik;  // 1/alpha = 3 / (2 beta k)
      const int ntries = REPEAT ? uc.max_tries : 1;
#pragma unroll 1
      for (int tr = 0; tr < ntries && !accepted; ++tr) {
        ++cnt.proposed;
        accepted = fx_propose(fx_draw_at(s, mu, sub, tr, t, key), inv_alpha, a);
      }
    } else {
      ++cnt.proposed;  // k = 0: degenerate staple (measure zero), leave the subgroup
    }
    if (accepted) {
      ++cnt.accepted;
      cfx R00, R01;
      fx_rotation(a, v, R00, R01);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        cfx x = cfx_of(us[0][c]), y = cfx_of(us[1][c]);
        fx_rotate_column(R00, R01, x, y);
        us[0][c] = cfx_short(x);
        us[1][c] = cfx_short(y);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const bool first = sub == 0;
      const cfxs x[3] = {us[0][c], us[1][c], us[2][c]}, y[3] = {A[c][0], A[c][1], A[c][2]};
      us[0][c] = first ? x[0] : x[2];
      us[1][c] = first ? x[2] : x[1];
      us[2][c] = first ? x[1] : x[0];
      A[c][0] = first ? y[0] : y[2];
      A[c][1] = first ? y[2] : y[1];
      A[c][2] = first ? y[1] : y[0];
    }
  }
  // after the last change: (row 0, row 2, row 1)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    u.e[0][c] = cfx_of(us[0][c]);
    u.e[1][c] = cfx_of(us[2][c]);
  }
  mat3<double> out;
  if (fx_reunitarise(u)) {
    fx_complete_row2(u);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) out.e[i][k] = mk(fx_to_double(u.e[i][k].re), fx_to_double(u.e[i][k].im));
  } else {  // a link of a configuration that was set with less than FP64 accuracy
    cx<double> r0[3], r1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      r0[k] = mk(fx_to_double(u.e[0][k].re), fx_to_double(u.e[0][k].im));
      r1[k] = mk(fx_to_double(u.e[1][k].re), fx_to_double(u.e[1][k].im));
    }
    gram_schmidt_rows01(r0, r1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      out.e[0][k] = r0[k];
      out.e[1][k] = r1[k];
    }
    complete_row2(out);
    if (MEAS) {
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k)
          u.e[i][k] = cfx{fx_from_double(out.e[i][k].re), fx_from_double(out.e[i][k].im)};
    }
  }
  store_f64(U, mu, p, h, g.Vh, out);
  if (MEAS) {
    facc tr{0, 0.0f};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        fx_mac(tr, u.e[i][k].re, Apart.e[k][i].re);
        fx_msub(tr, u.e[i][k].im, Apart.e[k][i].im);
      }
    *meas = (double)fx_merge_wide(tr) * (0x1p-58 / 3.0);
  }
  return cnt;
}

// ---------------------------------------------------------------------------
// The same update shared by LPL = 4 or 8 neighbouring lanes of a warp, for
// lattices whose half-sweep leaves the GPU mostly idle: there the time is the
// latency of one update.
//   staple: 4 lanes: lanes 0-2 take the two paths of one direction each; 8 lanes:
//     lanes 0-5 take one path each.  The paths are added as integers.
//   heatbath: lane c < 3 holds column c of the link and row c of the staple; the
//     projections and the Gram-Schmidt sums add up over the lanes as integers,
//     the scalars of a subgroup are computed by every lane.
//   draws: lane n < 3 draws the numbers of subgroup n, before it waits for the
//     half-sweep before this one (grid_wait), on which they do not depend.
// Integer sums make every link bit for bit that of update_link_f64.  All lanes
// of the warp call (shuffles); a group with active = false discards its
// result.
// ---------------------------------------------------------------------------
template <int LPL>
struct LaneGroup {
  int part, c, base;
  __device__ __forceinline__ LaneGroup() {
    const int lane = (int)threadIdx.x & 31;
    part = lane & (LPL - 1);
    c = part < 3 ? part : 0;
    base = lane & ~(LPL - 1);
  }
  // column c + s (mod 3)
  __device__ __forceinline__ int col(int s) const {
    const int k = c + s;
    return k >= 3 ? k - 3 : k;
  }
  template <typename T>
  __device__ __forceinline__ T from(T v, int k) const {
    return __shfl_sync(0xffffffffu, v, base + k);
  }
  __device__ __forceinline__ fx from(const fx& v, int k) const { return fx_make(from(v.h, k), from(v.l, k)); }
  __device__ __forceinline__ cfx from(const cfx& v, int k) const { return cfx{from(v.re, k), from(v.im, k)}; }
  // sum over the columns
  __device__ __forceinline__ long long sum(long long v) const { return v + from(v, col(1)) + from(v, col(2)); }
};

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <int LPL, bool REPEAT, typename KEY, typename G>
__device__ __forceinline__ UpdateCount update_link_f64_lanes(const G& g, double2* U, int h, int p, int mu,
                                                             const uint64_t* sweep, const KEY& key,
                                                             const UpdateConsts& uc, bool active) {
  const LaneGroup<LPL> lg;
  const uint64_t t = *sweep;
  const auto st = site_of(g, h, p);
  const uint32_t s = (uint32_t)canon(g, st);
  const fx_drawn mine = fx_draw_at(s, mu, lg.c, 0, t, key);
  UpdateCount cnt{0, 0};
  grid_wait();
  if (*(volatile const int*)uc.far) {  // links far from SU(3): one lane per link
    if (lg.part == 0 && active) cnt = update_link_f64_far(g, U, h, p, mu, t, key, uc, nullptr);
    return cnt;
  }
  h = store_index(g, st, h);
  const FxLink own(U, mu, p, h, g.Vh);
  const double2 mine_u[3] = {__ldcg(own.at(0, lg.c)), __ldcg(own.at(1, lg.c)), __ldcg(own.at(2, lg.c))};
  fx_staple A;
  fx_staple_zero(A);
  constexpr int kPaths = LPL == 8 ? 1 : 2;  // per lane
  if (lg.part * kPaths < 6)
    staple_paths_fx(A, g, U, st, h, p, mu, lg.part * kPaths, (lg.part + 1) * kPaths, FxRing(), nullptr);
  if constexpr (LPL == 8) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int q = 0; q < 2; ++q) A.r[i][k][q] += __shfl_down_sync(0xffffffffu, A.r[i][k][q], 3, LPL);
  }
  // row c of the sum: lane c + n (mod 3) sends its row c
  cfx a[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    long long m[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const long long x0 = A.r[0][k][q], x1 = A.r[1][k][q], x2 = A.r[2][k][q];
      m[q] = lg.c == 0 ? x0 : (lg.c == 1 ? x1 : x2);
      m[q] += lg.from(lg.c == 0 ? x2 : (lg.c == 1 ? x0 : x1), lg.col(1));  // row c - 1 goes to lane c - 1
      m[q] += lg.from(lg.c == 0 ? x1 : (lg.c == 1 ? x2 : x0), lg.col(2));
    }
    a[k] = cfx{fx_staple_entry(m[0], lg.c, 6), fx_staple_entry(m[1], lg.c, 6)};
  }
  cfx u[3] = {fx_entry(mine_u[0], 0u), fx_entry(mine_u[1], 0u), fx_entry(mine_u[2], 0u)};
#pragma unroll 1
  for (int sub = 0; sub < 3; ++sub) {
    long long r[4];
    fx_projection_column(u[0], u[1], a[0], a[1], r);
#pragma unroll
    for (int n = 0; n < 4; ++n) r[n] = lg.sum(r[n]);
    fx_drawn w;
    w.S = lg.from(mine.S, sub);
    w.u3 = lg.from(mine.u3, sub);
#pragma unroll
    for (int n = 0; n < 3; ++n) w.d[n] = lg.from(mine.d[n], sub);
    fx v[4], q[4];
    double ik;
    bool accepted = false;
    if (fx_direction(r, v, &ik)) {
      const double inv_alpha = uc.three_over_beta_f64 * ik;
      ++cnt.proposed;
      accepted = fx_propose(w, inv_alpha, q);
      if (REPEAT) {
#pragma unroll 1
        for (int tr = 1; tr < uc.max_tries && !accepted; ++tr) {
          ++cnt.proposed;
          accepted = fx_propose(fx_draw_at(s, mu, sub, tr, t, key), inv_alpha, q);
        }
      }
    } else {
      ++cnt.proposed;
    }
    if (accepted) {
      ++cnt.accepted;
      cfx R00, R01;
      fx_rotation(q, v, R00, R01);
      fx_rotate_column(R00, R01, u[0], u[1]);
    }
    const bool first = sub == 0;
    const cfx x[3] = {u[0], u[1], u[2]}, y[3] = {a[0], a[1], a[2]};
    u[0] = first ? x[0] : x[2];
    u[1] = first ? x[2] : x[1];
    u[2] = first ? x[1] : x[0];
    a[0] = first ? y[0] : y[2];
    a[1] = first ? y[2] : y[1];
    a[2] = first ? y[1] : y[0];
  }
  cfx r0 = u[0], r1 = u[2];
  fx_gram gr = fx_gram_column(r0, r1);
  gr.n0 = lg.sum(gr.n0);
  gr.n1 = lg.sum(gr.n1);
  gr.dr = lg.sum(gr.dr);
  gr.di = lg.sum(gr.di);
  fx_gs co;
  const bool ok = fx_gs_coefficients(gr, co);
  cx<double> o[3];
  if (__any_sync(0xffffffffu, lg.part < 3 && !ok)) {  // as in heatbath_fx
    const double d[4] = {fx_to_double(r0.re), fx_to_double(r0.im), fx_to_double(r1.re), fx_to_double(r1.im)};
    cx<double> b0[3], b1[3];
    mat3<double> m;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      b0[k] = mk(lg.from(d[0], k), lg.from(d[1], k));
      b1[k] = mk(lg.from(d[2], k), lg.from(d[3], k));
    }
    gram_schmidt_rows01(b0, b1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m.e[0][k] = b0[k];
      m.e[1][k] = b1[k];
    }
    complete_row2(m);
#pragma unroll
    for (int i = 0; i < 3; ++i) o[i] = lg.c == 0 ? m.e[i][0] : (lg.c == 1 ? m.e[i][1] : m.e[i][2]);
  }
  fx_gs_column(co, r0, r1);
  const cfx row2 = fx_row2_entry(lg.from(r0, lg.col(1)), lg.from(r0, lg.col(2)), lg.from(r1, lg.col(1)), lg.from(r1, lg.col(2)));
  if (ok) {
    o[0] = mk(fx_to_double(r0.re), fx_to_double(r0.im));
    o[1] = mk(fx_to_double(r1.re), fx_to_double(r1.im));
    o[2] = mk(fx_to_double(row2.re), fx_to_double(row2.im));
  }
  if (active && lg.part < 3 && link_ok(mu, p, h, g.Vh)) {
    double2* b = U + link_base(mu, p, g.Vh, kEntriesF64) + h + (size_t)lg.c * g.Vh;
#pragma unroll
    for (int i = 0; i < 3; ++i) b[(size_t)(3 * i) * g.Vh] = make_double2(o[i].re, o[i].im);
  }
  if (lg.part != 0 || !active) cnt = UpdateCount{0, 0};
  return cnt;
}

// One update of an FP64 store's link U_mu(x) (h, parity p as in site_of).
template <bool REPEAT, bool MEAS = false, typename KEY, typename G>
__device__ __forceinline__ UpdateCount update_link_f64(const G& g, double2* U, int h, int p, int mu, uint64_t t,
                                                       const KEY& key, const UpdateConsts& uc, double* meas = nullptr) {
  if (*(volatile const int*)uc.far) return update_link_f64_far(g, U, h, p, mu, t, key, uc, MEAS ? meas : nullptr);
  const auto st = site_of(g, h, p);
  const uint32_t s = (uint32_t)canon(g, st);
  h = store_index(g, st, h);
  fx_mat Apart;
  fx_staple A;
  fx_staple_zero(A);
  const FxRing ring;
  const FxLink own(U, mu, p, h, g.Vh);
  staple_paths_fx(A, g, U, st, h, p, mu, 0, 6, ring, &own, MEAS ? &Apart : nullptr);
  cp_async_wait<0>();
  fx_mat u;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) u.e[i][k] = fx_entry(ring.yz[3 * i + k], 0u);
  return heatbath_fx<REPEAT, MEAS>(g, U, h, p, mu, t, s, key, uc, u, fx_staple_mat(A, 6), Apart, meas);
}

// ---------------------------------------------------------------------------
// FP32-mixed staple on row pairs (su3_pair.cuh): every three-link path is an
// SU(3) matrix, so rows 0,1 are multiplied out two rows at a time and row 2
// is completed.
// ---------------------------------------------------------------------------
// The two paths of direction nu on row pairs, rows 0,1 (as forward_path and
// backward_path above), added to the staple in the same order.
template <bool CG, bool PAIRS = false, typename G>
__device__ __forceinline__ pm3 forward_path_p(const G& g, const float4* U, int h, int p, int mu, int nu, int h_pmu,
                                              int h_pnu) {
  const int q = p ^ 1;
  const pm3 a = load_pm3_l<CG, PAIRS>(U, nu, q, h_pmu, g.Vh);  // U_nu(x+mu)
  pm3 b = load_pm3_l<CG, PAIRS>(U, mu, q, h_pnu, g.Vh);        // U_mu(x+nu)
  complete_row2_p(b);
  pm3 t;
  mul_nd_p(a, b, t);
  pm3 c = load_pm3_l<CG, PAIRS>(U, nu, p, h, g.Vh);  // U_nu(x)
  complete_row2_p(c);
  pm3 f;
  mul_nd_p(t, c, f);
  return f;
}

template <bool CG, bool PAIRS = false, typename G>
__device__ __forceinline__ pm3 backward_path_p(const G& g, const float4* U, int p, int mu, int nu, int h_mnu,
                                               int h_pmu_mnu) {
  const int q = p ^ 1;
  pm3 d = load_pm3_l<CG, PAIRS>(U, nu, p, h_pmu_mnu, g.Vh);  // U_nu(x+mu-nu)
  complete_row2_p(d);
  const pm3 e = load_pm3_l<CG, PAIRS>(U, mu, q, h_mnu, g.Vh);  // U_mu(x-nu)
  pm3 hm;
  mul_nn_p(e, d, hm);
  complete_row2_p(hm);
  pm3 f = load_pm3_l<CG, PAIRS>(U, nu, q, h_mnu, g.Vh);  // U_nu(x-nu)
  complete_row2_p(f);
  pm3 b;
  mul_dn_p(hm, f, b);
  return b;
}

// A = F (rows 0,1 given, row 2 completed): the first term of a staple.
__device__ __forceinline__ void init_completed_p(pm3& A, const pm3& F) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    A.re[k] = F.re[k];
    A.im[k] = F.im[k];
  }
  complete_row2_p(A);
}

template <int MU, bool CG, bool PAIRS = false, typename G, typename S>
__device__ __forceinline__ pm3 staple_p(const G& g, const float4* U, const S& st, int h, int p,
                                        pm3* Apart = nullptr) {
  pm3 A;
  const int h_pmu = nb_half(g, st, MU, +1);
#pragma unroll
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == MU) continue;
    const int h_pnu = nb_half(g, st, nu, +1);
    const int h_mnu = nb_half(g, st, nu, -1);
    const int h_pmu_mnu = nb_half2(g, st, MU, nu);
    const pm3 F = forward_path_p<CG, PAIRS>(g, U, h, p, MU, nu, h_pmu, h_pnu);
    if (nu == (MU == 0 ? 1 : 0)) {
      init_completed_p(A, F);
    } else {
      acc_completed_p(A, F);
    }
    acc_completed_p(A, backward_path_p<CG, PAIRS>(g, U, p, MU, nu, h_mnu, h_pmu_mnu));
    if (Apart && nu == MU - 1) *Apart = A;
  }
  return A;
}

// The hardware square root (about 1 ulp): the FP32 heatbath needs no
// correctly rounded one.
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------------------
// One FP32-mixed link update: FP32 storage (rows 0,1), FP32 staple and
// heatbath, Gram-Schmidt coefficients in FP64 (EFT = false) or as
// compensated FP32 sums of FP64-class accuracy (EFT = true).  REPEAT = false
// compiles the one-hit heatbath without the retry loop.
// ---------------------------------------------------------------------------
template <int MU, bool CG, bool EFT, bool REPEAT, bool MEAS, typename KEY, typename G>
__device__ __forceinline__ UpdateCount heatbath_f32(const G& g, float4* U, int h, int p, uint64_t t, uint32_t s,
                                                    const KEY& key, const UpdateConsts& uc, const pm3& A,
                                                    const pm3& Apart, double* meas);

template <int MU, bool CG, bool EFT, bool REPEAT, bool MEAS = false, typename KEY, typename G>
__device__ __forceinline__ UpdateCount update_link_f32(const G& g, float4* U, int h, int p, uint64_t t,
                                                       const KEY& key, const UpdateConsts& uc, double* meas = nullptr) {
  const auto st = site_of(g, h, p);
  const uint32_t s = (uint32_t)canon(g, st);
  h = store_index(g, st, h);
  pm3 Apart;
  const pm3 A = staple_p<MU, CG>(g, U, st, h, p, MEAS ? &Apart : nullptr);
  return heatbath_f32<MU, CG, EFT, REPEAT, MEAS>(g, U, h, p, t, s, key, uc, A, Apart, meas);
}

// Everything after the staple (FP32 storage): three SU(2) heatbath steps,
// reunitarisation, store.
// The part of an FP32 proposal that does not depend on the staple.
struct DrawF32 {
  float L;                     // ln u0 + cos^2(2 pi u1) ln u2
  float u3, ct, sn, sphi, cphi;  // cos and sin of theta, sin and cos of phi - pi
};
template <int MU, typename KEY>
__device__ __forceinline__ DrawF32 draw_f32(uint32_t s, int sub, int tr, uint64_t t, const KEY& key) {
  const uint32_t w1b = (uint32_t)(MU | (sub << 2)) | ((uint32_t)tr << 6);
  const uint4 w0 = philox4x32_10(rng_counter(s, w1b, t, kTagUpdate), key);
  const uint4 w1 = philox4x32_10(rng_counter(s, w1b | (1u << 4), t, kTagUpdate), key);
  const float u0 = u01_f32(w0.x), u1 = u01_f32(w0.y), u2 = u01_f32(w0.z), u4 = u01_f32(w1.x), u5 = u01_f32(w1.y);
  const float cc = __cosf(fmaf(6.2831853f, u1, -3.14159265f));  // -cos(2 pi u1); only its square is used
  DrawF32 d;
  d.L = __fmaf_rn(__fmul_rn(cc, cc), __logf(u2), __logf(u0));
  d.u3 = u01_f32(w0.w);
  d.ct = __fmaf_rn(-2.0f, u4, 1.0f);
  d.sn = 2.0f * sqrt_approx(u4 * (1.0f - u4));  // sqrt(1 - ct^2)
  __sincosf(fmaf(6.2831853f, u5, -3.14159265f), &d.sphi, &d.cphi);  // angle 2 pi u5 - pi
  return d;
}

template <int MU, bool EFT, bool REPEAT, bool MEAS, bool PAIRS = false, bool DRAWN = false, typename KEY, typename G>
__device__ __forceinline__ UpdateCount heatbath_f32_on(const G& g, float4* U, int h, int p, uint64_t t, uint32_t s,
                                                       const KEY& key, const UpdateConsts& uc, const pm3& A,
                                                       const pm3& Apart, double* meas, pm3 u, bool store,
                                                       const DrawF32* drawn = nullptr);

template <int MU, bool CG, bool EFT, bool REPEAT, bool MEAS, typename KEY, typename G>
__device__ __forceinline__ UpdateCount heatbath_f32(const G& g, float4* U, int h, int p, uint64_t t, uint32_t s,
                                                    const KEY& key, const UpdateConsts& uc, const pm3& A,
                                                    const pm3& Apart, double* meas) {
  return heatbath_f32_on<MU, EFT, REPEAT, MEAS>(g, U, h, p, t, s, key, uc, A, Apart, meas,
                                                 load_pm3<CG>(U, MU, p, h, g.Vh), true);
}

// The same with the link's own rows 0,1 given (u); store = false computes
// everything but writes nothing (a lane that only keeps its warp converged).
// DRAWN: the first proposals' draws are given.
template <int MU, bool EFT, bool REPEAT, bool MEAS, bool PAIRS, bool DRAWN, typename KEY, typename G>
__device__ __forceinline__ UpdateCount heatbath_f32_on(const G& g, float4* U, int h, int p, uint64_t t, uint32_t s,
                                                       const KEY& key, const UpdateConsts& uc, const pm3& A,
                                                       const pm3& Apart, double* meas, pm3 u, bool store,
                                                       const DrawF32* drawn) {
  UpdateCount cnt{0, 0};
  complete_row2_p(u);
  const float three_over_beta = uc.three_over_beta;
#pragma unroll
  for (int sub = 0; sub < 3; ++sub) {
    const int i = subrow_i(sub), j = subrow_j(sub);
    // 2x2 block (i, j) of W = U A
    cx<float> wii, wij, wji, wjj;
    if (sub == 0) {
      // rows 0 and 1 as one pair: (W_0b, W_1b) = sum_c (U_0c, U_1c) A_cb
      float2 wr[2], wi[2];
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        float2 zr = make_float2(0.f, 0.f), zi = zr;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float ar = pre(A, c, b), ai = pim(A, c, b);
          zr = fma2(u.re[c], bc2(ar), zr);
          zr = fma2(u.im[c], bc2(-ai), zr);
          zi = fma2(u.re[c], bc2(ai), zi);
          zi = fma2(u.im[c], bc2(ar), zi);
        }
        wr[b] = zr;
        wi[b] = zi;
      }
      wii = mk(wr[0].x, wi[0].x);
      wji = mk(wr[0].y, wi[0].y);
      wij = mk(wr[1].x, wi[1].x);
      wjj = mk(wr[1].y, wi[1].y);
    } else {
      wii = mk(0.f, 0.f);
      wij = wii;
      wji = wii;
      wjj = wii;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        wii = mac(wii, pget(u, i, c), pget(A, c, i));
        wij = mac(wij, pget(u, i, c), pget(A, c, j));
        wji = mac(wji, pget(u, j, c), pget(A, c, i));
        wjj = mac(wjj, pget(u, j, c), pget(A, c, j));
      }
    }
    // 2r, as in su2_projection
    const float r[4] = {wii.re + wjj.re, wij.im + wji.im, wij.re - wji.re, wii.im - wjj.im};
    const float kk = __fmaf_rn(r[3], r[3], __fmaf_rn(r[2], r[2], __fmaf_rn(r[1], r[1], __fmul_rn(r[0], r[0]))));  // (2k)^2
    if (!(kk > 4e-30f)) {  // degenerate staple (measure zero): leave the subgroup
      ++cnt.proposed;
      continue;
    }
    const float ik = rsqrtf(kk);             // 1 / (2k)
    const float ia = three_over_beta * ik;  // 1/alpha = 3 / (2 beta k)
    bool acc = false;
    float a[4];
    const int ntries = REPEAT ? uc.max_tries : 1;
    for (int tr = 0; tr < ntries; ++tr) {
      // (the draws as in draw_f32, but in the order in which they are used: drawn
      // whole before the accept test, 18 x 10 x 14 x 22 took 3 to 8 % longer)
      if constexpr (DRAWN) {
        const DrawF32& d = drawn[sub];
        ++cnt.proposed;
        const float delta = __fmul_rn(-d.L, ia);
        if (__fmul_rn(d.u3, d.u3) > __fmaf_rn(-0.5f, delta, 1.0f)) continue;
        const float rho = sqrt_approx(fmaxf(0.0f, delta * (2.0f - delta)));
        const float rs = -rho * d.sn;
        a[0] = 1.0f - delta;
        a[1] = rs * d.cphi;
        a[2] = rs * d.sphi;
        a[3] = rho * d.ct;
      } else {
        const uint32_t w1b = (uint32_t)(MU | (sub << 2)) | ((uint32_t)tr << 6);
        const uint4 w0 = philox4x32_10(rng_counter(s, w1b, t, kTagUpdate), key);
        const uint4 w1 = philox4x32_10(rng_counter(s, w1b | (1u << 4), t, kTagUpdate), key);
        ++cnt.proposed;
        const float u0 = u01_f32(w0.x), u1 = u01_f32(w0.y), u2 = u01_f32(w0.z), u3 = u01_f32(w0.w);
        const float cc = __cosf(fmaf(6.2831853f, u1, -3.14159265f));  // -cos(2 pi u1); only its square is used
        const float delta = __fmul_rn(-__fmaf_rn(__fmul_rn(cc, cc), __logf(u2), __logf(u0)), ia);
        if (__fmul_rn(u3, u3) > __fmaf_rn(-0.5f, delta, 1.0f)) continue;
        const float u4 = u01_f32(w1.x), u5 = u01_f32(w1.y);
        const float rho = sqrt_approx(fmaxf(0.0f, delta * (2.0f - delta)));  // sqrt(1 - a0^2)
        const float ct = __fmaf_rn(-2.0f, u4, 1.0f);
        const float sn = 2.0f * sqrt_approx(u4 * (1.0f - u4));  // sqrt(1 - ct^2)
        float sphi, cphi;
        __sincosf(fmaf(6.2831853f, u5, -3.14159265f), &sphi, &cphi);  // angle 2 pi u5 - pi
        const float rs = -rho * sn;                                     // undo the shift by pi
        a[0] = 1.0f - delta;
        a[1] = rs * cphi;
        a[2] = rs * sphi;
        a[3] = rho * ct;
      }
      acc = true;
      break;
    }
    if (!acc) continue;
    const float v[4] = {r[0] * ik, r[1] * ik, r[2] * ik, r[3] * ik};
    // R = Y V^+ with Y = m(a), V = m(v), m(q) = [[q0 + i q3, q2 + i q1], [-q2 + i q1, q0 - i q3]]
    const cx<float> y00 = mk(a[0], a[3]), y01 = mk(a[2], a[1]);
    const cx<float> v00 = mk(v[0], v[3]), v01 = mk(v[2], v[1]), v10 = mk(-v[2], v[1]), v11 = mk(v[0], -v[3]);
    const cx<float> R00 = mac_cb(mac_cb(mk(0.f, 0.f), y00, v00), y01, v01);
    const cx<float> R01 = mac_cb(mac_cb(mk(0.f, 0.f), y00, v10), y01, v11);
    const cx<float> R10 = mk(-R01.re, R01.im);  // R keeps the SU(2) form
    const cx<float> R11 = mk(R00.re, -R00.im);
    if (sub == 0) {
      rotate01_p(u, R00, R01, R10, R11);
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const cx<float> ui = pget(u, i, c), uj = pget(u, j, c);
        pset(u, i, c, mac(mul(R00, ui), R01, uj));
        // row 2 leaves the last subgroup unused: reunitarisation rebuilds it
        if (sub < 2) pset(u, j, c, mac(mul(R10, ui), R11, uj));
      }
    }
    ++cnt.accepted;
  }
  cx<float> r0[3], r1[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r0[k] = pget(u, 0, k);
    r1[k] = pget(u, 1, k);
  }
  float o[12];
  reunitarise_f32<EFT>(r0, r1, o);
  if (store) {
    if (PAIRS)
      store_pair_site(U, MU, p, h, g.Vh / 2, o);
    else
      store_f32_rows01(U, MU, p, h, g.Vh, o);
  }
  if (MEAS) {
    // the stored link, row 2 completed, against A_<
    mat3<float> un;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      un.e[0][k] = mk(o[2 * k], o[2 * k + 1]);
      un.e[1][k] = mk(o[6 + 2 * k], o[6 + 2 * k + 1]);
    }
    complete_row2(un);
    float tr = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const cx<float> ak = pget(Apart, k, i);
        tr = fmaf(un.e[i][k].re, ak.re, fmaf(-un.e[i][k].im, ak.im, tr));
      }
    *meas = (double)tr * (1.0 / 3.0);
  }
  return cnt;
}

}  // namespace su3dev
