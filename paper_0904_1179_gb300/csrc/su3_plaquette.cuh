// su3_plaquette.cuh -- the mean plaquette of a link store: per-block sums of Re Tr
// U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+ over sites and planes, added up in a
// fixed order.  Shared by the kernels of single lattices and of batches.
#pragma once

#include "su3_device.cuh"
#include "su3_sitepair.cuh"
#include "su3_update.cuh"

namespace su3dev {

constexpr int kPlaqThreads = 256;
__host__ __device__ inline int plaq_blocks(const Geometry& g) { return (2 * g.Vh + kPlaqThreads - 1) / kPlaqThreads; }

template <typename T>
__device__ __forceinline__ mat3<T> load_any(const void* U, int mu, int p, int h, int Vh, bool pairs);
template <>
__device__ __forceinline__ mat3<double> load_any<double>(const void* U, int mu, int p, int h, int Vh, bool) {
  return load_f64((const double2*)U, mu, p, h, Vh);
}
template <>
__device__ __forceinline__ mat3<float> load_any<float>(const void* U, int mu, int p, int h, int Vh, bool pairs) {
  return load_f32_any((const float4*)U, mu, p, h, Vh, pairs);
}

// Re Tr(X Y^+) with X = U_mu(x) U_nu(x+mu), Y = U_nu(x) U_mu(x+nu).
template <typename T>
__device__ __forceinline__ double plaq_site(const Geometry& g, const void* U, const Site& st, int h, int p, bool pairs) {
  const int q = p ^ 1;
  double sum = 0.0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu)
#pragma unroll
    for (int nu = mu + 1; nu < 4; ++nu) {
      const mat3<T> a = load_any<T>(U, mu, p, h, g.Vh, pairs);
      const mat3<T> b = load_any<T>(U, nu, q, nb_half(g, st, mu, +1), g.Vh, pairs);
      const mat3<T> c = load_any<T>(U, nu, p, h, g.Vh, pairs);
      const mat3<T> d = load_any<T>(U, mu, q, nb_half(g, st, nu, +1), g.Vh, pairs);
      T tr = T(0);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          cx<T> x = mk(T(0), T(0)), y = x;
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            x = mac(x, a.e[i][j], b.e[j][k]);
            y = mac(y, c.e[i][j], d.e[j][k]);
          }
          tr = fma(x.re, y.re, tr);
          tr = fma(x.im, y.im, tr);
        }
      sum += (double)tr;
    }
  return sum;
}

// Sum over the block's threads (up to 32 warps) in thread 0 of warp 0.
__device__ __forceinline__ double plaq_block_sum(double v) {
  __shared__ double red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double w = 0.0;
  if (threadIdx.x < 32) {
    w = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  }
  return w;
}

// Block `block` of a lattice's partial sums: one thread per site, six planes,
// products in the storage precision, FP64 sums.
template <typename T>
__device__ __forceinline__ void plaq_block(const Geometry& g, const void* U, bool pairs, int block, double* out) {
  const int idx = block * (int)blockDim.x + (int)threadIdx.x;  // over 2 * Vh: (parity, h)
  double v = 0.0;
  if (idx < 2 * g.Vh) {
    const int p = idx >= g.Vh ? 1 : 0;
    const int h = idx - p * g.Vh;
    v = plaq_site<T>(g, U, site_of(g, h, p), h, p, pairs);
  }
  v = plaq_block_sum(v);
  if (threadIdx.x == 0) *out = v;
}

// One block: out = scale * sum of n partials.
__device__ __forceinline__ void sum_partials(const double* partials, int n, double scale, double* out) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += partials[i];
  v = plaq_block_sum(v);
  if (threadIdx.x == 0) *out = v * scale;
}

// ---------------------------------------------------------------------------
// FP64 stores, in the arithmetic of su3_fx.cuh: a block takes groups of 32 sites,
// its six warps the six planes.  (One thread per site on the FP64 pipe took 2.51
// ms at 32^4 and, a serial chain of 1,300 FP64 FMAs, 111 us at 4^4.)
// ---------------------------------------------------------------------------
constexpr int kPlaqFxThreads = 192;
constexpr int kPlaqFxSites = 32;
// Groups per block: one, more where that made over 16384 blocks.
__host__ __device__ inline int plaq_fx_groups(const Geometry& g) { return (2 * g.Vh + kPlaqFxSites - 1) / kPlaqFxSites; }
__host__ __device__ inline int plaq_fx_passes(const Geometry& g) { return (plaq_fx_groups(g) + 16383) / 16384; }
__host__ __device__ inline int plaq_fx_blocks(const Geometry& g) {
  return (plaq_fx_groups(g) + plaq_fx_passes(g) - 1) / plaq_fx_passes(g);
}

// Re Tr (a b)(c d)^+, a = U_mu(x), b = U_nu(x+mu), c = U_nu(x), d = U_mu(x+nu), in units
// of 2^-60.
__device__ __forceinline__ long long plaq_plane_fx(const Geometry& g, const void* U, const Site& st, int h, int p, int mu,
                                                   int nu) {
  const int q = p ^ 1;
  const FxLink A(U, mu, p, h, g.Vh), B(U, nu, q, nb_half_rt(g, st, mu, +1), g.Vh), C(U, nu, p, h, g.Vh),
      D(U, mu, q, nb_half_rt(g, st, nu, +1), g.Vh);
  cfx a[3][3], c[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[i][k] = fx_entry(__ldg(A.at(i, k)), 0u);
      c[i][k] = fx_entry(__ldg(C.at(i, k)), 0u);
    }
  long long tr = 0;
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    cfx b[3], d[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      b[j] = fx_entry(__ldg(B.at(j, k)), 0u);
      d[j] = fx_entry(__ldg(D.at(j, k)), 0u);
    }
    facc s{0, 0.0f};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      cfacc x = cfx_zero(), y = cfx_zero();
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cfx_mac(x, a[i][j], b[j]);
        cfx_mac(y, c[i][j], d[j]);
      }
      const cfx u = cfx_norm(x), v = cfx_norm(y);
      fx_mac(s, u.re, v.re);
      fx_mac(s, u.im, v.im);
    }
    tr += fx_merge(s);
  }
  return tr;
}

// The same in FP64 arithmetic, for configurations with links far from SU(3).
static __device__ __noinline__ double plaq_plane_far(const Geometry& g, const void* U, const Site& st, int h, int p, int mu,
                                              int nu) {
  const int q = p ^ 1;
  const mat3<double> a = load_f64((const double2*)U, mu, p, h, g.Vh), c = load_f64((const double2*)U, nu, p, h, g.Vh);
  const mat3<double> b = load_f64((const double2*)U, nu, q, nb_half_rt(g, st, mu, +1), g.Vh);
  const mat3<double> d = load_f64((const double2*)U, mu, q, nb_half_rt(g, st, nu, +1), g.Vh);
  double tr = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cx<double> x = mk(0.0, 0.0), y = x;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        x = mac(x, a.e[i][j], b.e[j][k]);
        y = mac(y, c.e[i][j], d.e[j][k]);
      }
      tr = fma(x.im, y.im, fma(x.re, y.re, tr));
    }
  return tr;
}

__device__ __forceinline__ void plaq_block_fx(const Geometry& g, const void* U, const int* far, int block, double* out) {
  const int plane = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  const int mu = plane < 3 ? 0 : (plane < 5 ? 1 : 2), nu = plane < 3 ? plane + 1 : (plane < 5 ? plane - 1 : 3);
  const int passes = plaq_fx_passes(g);
  const bool f = *far != 0;
  double v = 0.0;
#pragma unroll 1
  for (int n = 0; n < passes; ++n) {
    const long long idx = ((long long)block * passes + n) * kPlaqFxSites + lane;  // over 2 * Vh: (parity, h)
    if (idx < 2LL * g.Vh) {
      const int p = idx >= g.Vh ? 1 : 0;
      const int h = (int)(idx - (long long)p * g.Vh);
      const Site st = site_of(g, h, p);
      v += f ? plaq_plane_far(g, U, st, h, p, mu, nu) : (double)plaq_plane_fx(g, U, st, h, p, mu, nu) * 0x1p-60;
    }
  }
  v = plaq_block_sum(v);
  if (threadIdx.x == 0) *out = v;
}

}  // namespace su3dev
