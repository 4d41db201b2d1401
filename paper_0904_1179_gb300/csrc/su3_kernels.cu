// su3_kernels.cu -- sm_103a kernels of the checkerboard SU(3) heatbath sweep.
//
// One thread updates one link U_mu(x) of the half-sweep (mu, parity): it
// gathers the six-staple sum from the 18 neighbouring links, runs the one-hit
// Kennedy-Pendleton heatbath in the SU(2) subgroups (0,1), (0,2), (1,2)
// (Cabibbo-Marinari), reunitarises and stores the link.  Links of one
// (mu, parity) never enter each other's staples (checkerboard updating,
// Abstract and Sec. 1 of Berg & Wu, arXiv:0904.1179), so threads are
// independent; the counter-based Philox stream makes the result independent of
// the launch configuration.  The work is a 4D stencil of 3x3 complex products,
// not a dense contraction, so it runs on the CUDA cores.  The FP64 store's
// half-sweeps are in su3_kernels_f64.cu.
#include "su3_kernels.h"

#include "su3_device.cuh"
#include "su3_plaquette.cuh"
#include "su3_reduce.cuh"
#include "su3_sitepair.cuh"
#include "su3_update.cuh"

using namespace su3dev;

// Register budget of the FP32 half-sweep: __launch_bounds__(threads, min blocks
// per SM), every block size up to kMaxSweepThreads legal.  Two blocks of 256
// (126 registers, no spills) instead of four (64 registers): GB300, ms per sweep,
// mixed and EFT: 18 x 10 x 14 x 22 0.0698 -> 0.0596 and 0.0593 -> 0.0475 (few
// warps: more loads in flight each), 30^4 0.4019 -> 0.4026 and 0.385 -> 0.356, 42^4
// 1.3681 -> 1.3694 and 1.324 -> 1.244; mixed 26^4 0.242 -> 0.229, 36^3 x 30 0.653 ->
// 0.648, 50^4 2.703 -> 2.692, but 42 x 30 x 44 x 22 0.5744 -> 0.5758: EFT gains
// throughout, mixed up to about 0.25 % less on large lattices of some shapes and up
// to 5 % more on others, which no rule on the size tells apart.
#ifndef SU3_F32_LB_THREADS
#define SU3_F32_LB_THREADS kMaxSweepThreads
#endif
#ifndef SU3_F32_MINBLOCKS
#define SU3_F32_MINBLOCKS 2
#endif

namespace {

// ---------------------------------------------------------------------------
// Single-lattice half-sweeps: one thread per link of (mu, parity).
// ---------------------------------------------------------------------------
// Four lanes per link for FP32 storage (small lattices): lanes 0-2 form the two
// paths of one direction each; rows 0,1 of the paths on row pairs (12 floats
// each) are gathered into lane 0 and added in the single-thread order, and the random numbers of the three subgroups are drawn
// side by side; no register cap (small lattices leave the SMs nearly empty).
__device__ __forceinline__ pm3 shfl_pm3_rows01(const pm3& m, int src) {
  pm3 r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.re[k].x = __shfl_sync(0xffffffffu, m.re[k].x, src);
    r.re[k].y = __shfl_sync(0xffffffffu, m.re[k].y, src);
    r.im[k].x = __shfl_sync(0xffffffffu, m.im[k].x, src);
    r.im[k].y = __shfl_sync(0xffffffffu, m.im[k].y, src);
  }
  return r;
}

__device__ __forceinline__ DrawF32 shfl_draw(const DrawF32& d, int src) {
  return DrawF32{__shfl_sync(0xffffffffu, d.L, src),    __shfl_sync(0xffffffffu, d.u3, src),
                 __shfl_sync(0xffffffffu, d.ct, src),   __shfl_sync(0xffffffffu, d.sn, src),
                 __shfl_sync(0xffffffffu, d.sphi, src), __shfl_sync(0xffffffffu, d.cphi, src)};
}

template <int MU, bool STATS, bool EFT, bool PAIRS>
__global__ void __launch_bounds__(kMaxSweepThreads) k_half_sweep_f32_split(HalfSweepArgs args) {
  const Geometry& g = args.geom;
  const int p = args.parity;
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  const int link = gid >> 2, part = gid & 3;
  const bool active = link < g.Vh;
  const int h = active ? link : 0;
  const Site st = site_of(g, h, p);
  float4* U = (float4*)args.links;
  pm3 F = zero_p(), B = zero_p();
  if (part < 3) {
    const int nu = part < MU ? part : part + 1;
    const int h_pmu = nb_half(g, st, MU, +1);
    F = forward_path_p<false, PAIRS>(g, U, h, p, MU, nu, h_pmu, nb_half_rt(g, st, nu, +1));
    B = backward_path_p<false, PAIRS>(g, U, p, MU, nu, nb_half_rt(g, st, nu, -1), nb_half2_rt(g, st, MU, nu));
  }
  const int lane0 = (threadIdx.x & 31) & ~3;
  // lane n < 3 draws subgroup n's numbers; lane 0 uses them all
  const uint32_t s = (uint32_t)canon(g, st);
  const DrawF32 mine = draw_f32<MU>(s, part < 3 ? part : 0, 0, *args.sweep, args.key);
  DrawF32 draws[3];
#pragma unroll
  for (int n = 0; n < 3; ++n) draws[n] = shfl_draw(mine, lane0 + n);
  pm3 A;
  init_completed_p(A, F);
  acc_completed_p(A, B);
#pragma unroll
  for (int k = 1; k < 3; ++k) {
    acc_completed_p(A, shfl_pm3_rows01(F, lane0 + k));
    acc_completed_p(A, shfl_pm3_rows01(B, lane0 + k));
  }
  UpdateCount c{0, 0};
  if (part == 0 && active) {
    const UpdateConsts uc{args.three_over_beta_f64, args.three_over_beta, 1, sweep_far(args.sweep)};
    c = heatbath_f32_on<MU, EFT, false, false, PAIRS, true>(g, U, h, p, *args.sweep, s, args.key, uc, A, A, nullptr,
                                                             load_pm3_l<false, PAIRS>(U, MU, p, h, g.Vh), true, draws);
  }
  count_stats<STATS>(c, args.stats);
}

// One thread per link of a site-paired store (small lattices).
template <int MU, bool STATS, bool EFT>
__global__ void __launch_bounds__(SU3_F32_LB_THREADS, SU3_F32_MINBLOCKS) k_half_sweep_f32_single(HalfSweepArgs args) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  UpdateCount c{0, 0};
  if (h < args.geom.Vh) {
    const Geometry& g = args.geom;
    const UpdateConsts uc{args.three_over_beta_f64, args.three_over_beta, 1, nullptr};
    float4* U = (float4*)args.links;
    const Site st = site_of(g, h, args.parity);
    const pm3 A = staple_p<MU, false, true>(g, U, st, h, args.parity);
    c = heatbath_f32_on<MU, EFT, false, false, true>(g, U, h, args.parity, *args.sweep, (uint32_t)canon(g, st), args.key,
                                                     uc, A, A, nullptr,
                                                     load_pm3_l<false, true>(U, MU, args.parity, h, g.Vh), true);
  }
  count_stats<STATS>(c, args.stats);
}

template <int MU, bool STATS, bool EFT, bool REPEAT, bool MEAS>
__global__ void __launch_bounds__(SU3_F32_LB_THREADS, SU3_F32_MINBLOCKS) k_half_sweep_f32(HalfSweepArgs args) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  UpdateCount c{0, 0};
  double m = 0.0;
  if (h < args.geom.Vh) {
    const UpdateConsts uc{args.three_over_beta_f64, args.three_over_beta, args.max_tries, sweep_far(args.sweep)};
    c = update_link_f32<MU, false, EFT, REPEAT, MEAS>(args.geom, (float4*)args.links, h, args.parity, *args.sweep,
                                                      args.key, uc, &m);
  }
  count_stats<STATS>(c, args.stats);
  if (MEAS) block_partial(m, args.meas);
}

// far: nfar pairs of flags (far and far_next of SweepState).
__global__ void k_increment(uint64_t* counter, uint64_t n, int* far, int nfar) {
  if (threadIdx.x == 0) *counter += n;
  for (int i = threadIdx.x; i < nfar; i += blockDim.x) {
    far[2 * i] = far[2 * i + 1];
    far[2 * i + 1] = 0;
  }
}

__global__ void __launch_bounds__(1024) k_meas_final(const double* parts, int n, double scale, const uint64_t* sweep,
                                                     double* out, int cap) {
  __shared__ double red[32];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += parts[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double w = threadIdx.x < (int)(blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (threadIdx.x == 0) out[*sweep % (uint64_t)cap] = w * scale;
  }
}
__global__ void k_set_counter(uint64_t* counter, uint64_t n) { *counter = n; }

// ---------------------------------------------------------------------------
// Start configurations.
// ---------------------------------------------------------------------------
__global__ void k_cold_start(InitArgs args) {
  const Geometry g = args.geom;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;  // over 8 * Vh (mu, parity, h)
  if (idx >= 8 * g.Vh) return;
  const int mp = idx / g.Vh, h = idx - mp * g.Vh;
  const int mu = mp >> 1, p = mp & 1;
  if (args.precision == 0) {
    mat3<double> m = zero3<double>();
    m.e[0][0] = m.e[1][1] = m.e[2][2] = mk(1.0, 0.0);
    store_f64((double2*)args.links, mu, p, h, g.Vh, m);
  } else {
    float o[12] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f};
    store_f32_rows01_any((float4*)args.links, mu, p, h, g.Vh, args.pairs, o);
  }
}

// Haar SU(3): two complex Gaussian rows (Box-Muller on Philox tag 1 words,
// counter (s, mu | call<<4, 0, 1), call = 0..5), Gram-Schmidt, row 2 completed.
__global__ void k_hot_start(InitArgs args) {
  const Geometry g = args.geom;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 8 * g.Vh) return;
  const int mp = idx / g.Vh, h = idx - mp * g.Vh;
  const int mu = mp >> 1, p = mp & 1;
  const Site st = site_of(g, h, p);
  const uint32_t s = (uint32_t)canon(g, st);
  double gz[12];
#pragma unroll
  for (int call = 0; call < 6; ++call) {
    const uint4 w = philox4x32_10(rng_counter(s, (uint32_t)(mu | (call << 4)), 0, kTagHotStart), args.key);
    const double ua = u01_f64(w.x, w.y), ub = u01_f64(w.z, w.w);
    const double rad = sqrt(-2.0 * log(ua));
    double sn, cs;
    sincos(kTwoPi * ub, &sn, &cs);
    gz[2 * call] = rad * cs;
    gz[2 * call + 1] = rad * sn;
  }
  cx<double> r0[3], r1[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r0[k] = mk(gz[2 * k], gz[2 * k + 1]);
    r1[k] = mk(gz[6 + 2 * k], gz[6 + 2 * k + 1]);
  }
  gram_schmidt_rows01(r0, r1);
  if (args.precision == 0) {
    mat3<double> m;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m.e[0][k] = r0[k];
      m.e[1][k] = r1[k];
    }
    complete_row2(m);
    store_f64((double2*)args.links, mu, p, h, g.Vh, m);
  } else {
    float o[12];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      o[2 * k] = (float)r0[k].re;
      o[2 * k + 1] = (float)r0[k].im;
      o[6 + 2 * k] = (float)r1[k].re;
      o[6 + 2 * k + 1] = (float)r1[k].im;
    }
    store_f32_rows01_any((float4*)args.links, mu, p, h, g.Vh, args.pairs, o);
  }
}

// ---------------------------------------------------------------------------
// Plaquette: one thread per site, six planes (su3_plaquette.cuh), fixed-order
// block reduction into partials[blockIdx.x], then one block sums the partials.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kPlaqThreads) k_plaquette_partial(PlaqArgs args) {
  plaq_block<T>(args.geom, args.links, args.pairs != 0, (int)blockIdx.x, args.partials + blockIdx.x);
}

__global__ void __launch_bounds__(1024) k_plaquette_final(const double* partials, int n, double scale, double* out) {
  sum_partials(partials, n, scale, out);
}

// ---------------------------------------------------------------------------
// Canonical host layout <-> device store, for a chunk of sites [s_begin, s_begin + n).
// Canonical: double[s][mu][row][col][re/im].
// ---------------------------------------------------------------------------
// Row 2 from FP32 rows 0,1 in FP64 with every product and sum rounded
// separately (no contraction): conj(row0 x row1).
__device__ __forceinline__ cx<double> cmul_rn(cx<double> a, cx<double> b) {
  return mk(__dsub_rn(__dmul_rn(a.re, b.re), __dmul_rn(a.im, b.im)), __dadd_rn(__dmul_rn(a.re, b.im), __dmul_rn(a.im, b.re)));
}

__global__ void k_canon_to_store(ConvArgs args) {
  const Geometry g = args.geom;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4LL * args.n_sites) return;
  const int mu = (int)(idx / args.n_sites);
  const long long i = idx - (long long)mu * args.n_sites;
  const long long s = args.s_begin + i;
  const int h = (int)(s >> 1);
  const int x0 = (int)(s % g.L0);
  const int r = (int)(s / g.L0);
  const int x1 = r % g.L1, x2 = (r / g.L1) % g.L2, x3 = r / (g.L1 * g.L2);
  const int p = (x0 + x1 + x2 + x3) & 1;
  const double* src = args.canon + (i * 4 + mu) * 18;
  if (args.precision == 0) {
    mat3<double> m;
#pragma unroll
    for (int c = 0; c < 9; ++c) m.e[c / 3][c % 3] = mk(src[2 * c], src[2 * c + 1]);
    if (far_from_su3(m)) {
      *(volatile int*)args.far = 1;
      if (args.far_host) *(volatile int*)args.far_host = 1;
    }
    store_f64((double2*)args.links, mu, p, h, g.Vh, m);
  } else {
    float o[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) o[c] = (float)src[c];
    store_f32_rows01_any((float4*)args.links, mu, p, h, g.Vh, args.pairs, o);
  }
}

// One block per tile of 32 sites, one thread per link; the tile's 576 B per site
// pass through shared memory so that they leave as whole 16-byte runs: the
// destination is the staging buffer or, for page-locked memory that the GPU
// addresses, the caller's buffer itself (su3_transfer), which is bound by the
// host link (193 GB/s for a kernel's stores and for the copy engine alike).
// 37 16-byte words a site, not 36: free of bank conflicts.
constexpr int kConvSites = 32, kConvWords = 37;
__global__ void __launch_bounds__(4 * kConvSites) k_store_to_canon(ConvArgs args) {
  __shared__ double2 tile[kConvSites * kConvWords];
  const Geometry g = args.geom;
  if (args.status && blockIdx.x == 0 && threadIdx.x == 0) *args.status_host = *args.status;
  const long long i0 = (long long)blockIdx.x * kConvSites;
  const int n = (int)(args.n_sites - i0 < kConvSites ? args.n_sites - i0 : kConvSites);  // sites of this tile
  const int mu = threadIdx.x / kConvSites, i = threadIdx.x % kConvSites;
  if (i < n) {
    const long long s = args.s_begin + i0 + i;
    const int h = (int)(s >> 1);
    const int x0 = (int)(s % g.L0);
    const int r = (int)(s / g.L0);
    const int x1 = r % g.L1, x2 = (r / g.L1) % g.L2, x3 = r / (g.L1 * g.L2);
    const int p = (x0 + x1 + x2 + x3) & 1;
    double2* dst = tile + i * kConvWords + mu * 9;
    if (args.precision == 0) {
      const mat3<double> m = load_f64((const double2*)args.links, mu, p, h, g.Vh);
#pragma unroll
      for (int c = 0; c < 9; ++c) dst[c] = make_double2(m.e[c / 3][c % 3].re, m.e[c / 3][c % 3].im);
    } else {
      const mat3<float> m = load_f32_rows01_any((const float4*)args.links, mu, p, h, g.Vh, args.pairs);
      cx<double> a[3], b[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        a[k] = mk((double)m.e[0][k].re, (double)m.e[0][k].im);
        b[k] = mk((double)m.e[1][k].re, (double)m.e[1][k].im);
        dst[k] = make_double2(a[k].re, a[k].im);
        dst[3 + k] = make_double2(b[k].re, b[k].im);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
        const cx<double> x = cmul_rn(a[k1], b[k2]), y = cmul_rn(a[k2], b[k1]);
        dst[6 + k] = make_double2(__dsub_rn(x.re, y.re), -__dsub_rn(x.im, y.im));
      }
    }
  }
  __syncthreads();
  double2* out = (double2*)args.canon + i0 * 36;
  for (int e = threadIdx.x; e < n * 36; e += 4 * kConvSites) out[e] = tile[e / 36 * kConvWords + e % 36];
}

}  // namespace

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
template <int MU, bool STATS, bool EFT, bool REPEAT, bool MEAS>
static cudaError_t launch_f32(const HalfSweepArgs& a, int blocks, int threads, cudaStream_t s) {
  k_half_sweep_f32<MU, STATS, EFT, REPEAT, MEAS><<<blocks, threads, 0, s>>>(a);
  return cudaGetLastError();
}

template <int MU, bool STATS, bool REPEAT, bool MEAS>
static cudaError_t launch_prec(const HalfSweepArgs& a, int precision, int blocks, int threads, cudaStream_t s) {
  if (precision == 2) return launch_f32<MU, STATS, true, REPEAT, MEAS>(a, blocks, threads, s);
  return launch_f32<MU, STATS, false, REPEAT, MEAS>(a, blocks, threads, s);
}

template <int MU, bool STATS, bool EFT>
static void launch_f32_split(const HalfSweepArgs& a, int blocks, int threads, cudaStream_t s) {
  if (a.pairs)
    k_half_sweep_f32_split<MU, STATS, EFT, true><<<blocks, threads, 0, s>>>(a);
  else
    k_half_sweep_f32_split<MU, STATS, EFT, false><<<blocks, threads, 0, s>>>(a);
}

template <int MU>
static cudaError_t launch_half_sweep_mu(const HalfSweepArgs& a, int precision, bool stats, int threads, cudaStream_t s) {
  const int blocks = (a.geom.Vh + threads - 1) / threads;
  const bool repeat = a.max_tries > 1;
  // FP32 in the site-paired layout: the paired kernel, except for the
  // four-lane form of small lattices
  if (precision != 0 && a.pairs && a.single && !a.split && !repeat && !(MU > 0 && a.meas)) {
    if (precision == 2) {
      if (stats)
        k_half_sweep_f32_single<MU, true, true><<<blocks, threads, 0, s>>>(a);
      else
        k_half_sweep_f32_single<MU, false, true><<<blocks, threads, 0, s>>>(a);
    } else {
      if (stats)
        k_half_sweep_f32_single<MU, true, false><<<blocks, threads, 0, s>>>(a);
      else
        k_half_sweep_f32_single<MU, false, false><<<blocks, threads, 0, s>>>(a);
    }
    return cudaGetLastError();
  }
  if (precision != 0 && a.pairs && !(a.split && !repeat && !(MU > 0 && a.meas)))
    return su3k_launch_half_sweep_pair(a, MU, precision == 2, stats, threads, s);
  if (MU > 0 && a.meas) {  // fused plaquette (statistics are not counted in these phases)
    return repeat ? launch_prec<MU, false, true, (MU > 0)>(a, precision, blocks, threads, s)
                  : launch_prec<MU, false, false, (MU > 0)>(a, precision, blocks, threads, s);
  }
  if (a.split && !repeat) {
    const int sblocks = (4 * a.geom.Vh + threads - 1) / threads;
    if (precision == 2) {
      if (stats)
        launch_f32_split<MU, true, true>(a, sblocks, threads, s);
      else
        launch_f32_split<MU, false, true>(a, sblocks, threads, s);
    } else {
      if (stats)
        launch_f32_split<MU, true, false>(a, sblocks, threads, s);
      else
        launch_f32_split<MU, false, false>(a, sblocks, threads, s);
    }
    return cudaGetLastError();
  }
  if (stats)
    return repeat ? launch_prec<MU, true, true, false>(a, precision, blocks, threads, s)
                  : launch_prec<MU, true, false, false>(a, precision, blocks, threads, s);
  return repeat ? launch_prec<MU, false, true, false>(a, precision, blocks, threads, s)
                : launch_prec<MU, false, false, false>(a, precision, blocks, threads, s);
}

cudaError_t su3k_launch_half_sweep(const HalfSweepArgs& a, int mu, int precision, bool stats, int threads, cudaStream_t s) {
  if (precision == 0) return su3k_launch_half_sweep_f64(a, mu, stats, threads, s);
  switch (mu) {
    case 0: return launch_half_sweep_mu<0>(a, precision, stats, threads, s);
    case 1: return launch_half_sweep_mu<1>(a, precision, stats, threads, s);
    case 2: return launch_half_sweep_mu<2>(a, precision, stats, threads, s);
    default: return launch_half_sweep_mu<3>(a, precision, stats, threads, s);
  }
}

SU3_BOUNDS_STATUS_FN(su3k_bounds_status_kernels)

int su3k_half_sweep_blocks(const HalfSweepArgs& a, int precision, int threads) {
  const int n = (precision != 0 && a.pairs) ? a.pgeom.Vh : a.geom.Vh;
  return (n + threads - 1) / threads;
}

cudaError_t su3k_launch_increment(uint64_t* counter, uint64_t n, int* far, int nfar, cudaStream_t s) {
  k_increment<<<1, nfar > 1 ? 128 : 1, 0, s>>>(counter, n, far, nfar);
  return cudaGetLastError();
}

cudaError_t su3k_launch_meas_final(const double* parts, int nparts, double scale, const uint64_t* sweep, double* out,
                                   int cap, cudaStream_t s) {
  k_meas_final<<<1, 1024, 0, s>>>(parts, nparts, scale, sweep, out, cap);
  return cudaGetLastError();
}

cudaError_t su3k_launch_set_counter(uint64_t* counter, uint64_t n, cudaStream_t s) {
  k_set_counter<<<1, 1, 0, s>>>(counter, n);
  return cudaGetLastError();
}

cudaError_t su3k_launch_init(const InitArgs& a, bool hot, cudaStream_t s) {
  const long long n = 8LL * a.geom.Vh;
  const int threads = 128;
  const int blocks = (int)((n + threads - 1) / threads);
  if (hot)
    k_hot_start<<<blocks, threads, 0, s>>>(a);
  else
    k_cold_start<<<blocks, threads, 0, s>>>(a);
  return cudaGetLastError();
}

int su3k_plaquette_blocks(const Geometry& g) { return plaq_blocks(g); }

cudaError_t su3k_launch_plaquette(const PlaqArgs& a, int precision, double* out, cudaStream_t s) {
  const int blocks = su3k_plaquette_blocks(a.geom);
  if (precision == 0)
    k_plaquette_partial<double><<<blocks, kPlaqThreads, 0, s>>>(a);
  else
    k_plaquette_partial<float><<<blocks, kPlaqThreads, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const double V = 2.0 * (double)a.geom.Vh;
  k_plaquette_final<<<1, 1024, 0, s>>>(a.partials, blocks, 1.0 / (3.0 * 6.0 * V), out);
  return cudaGetLastError();
}

cudaError_t su3k_launch_conv(const ConvArgs& a, bool to_store, cudaStream_t s) {
  const long long n = 4LL * a.n_sites;
  if (n == 0) return cudaSuccess;
  if (to_store)
    k_canon_to_store<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a);
  else
    k_store_to_canon<<<(unsigned)((a.n_sites + kConvSites - 1) / kConvSites), 4 * kConvSites, 0, s>>>(a);
  return cudaGetLastError();
}
