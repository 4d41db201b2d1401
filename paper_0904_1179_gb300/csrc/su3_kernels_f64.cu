// su3_kernels_f64.cu -- the half-sweeps of the FP64 store (see su3_kernels.cu):
// one thread per link, or four lanes per link on small lattices.  The update
// runs on the integer and FP32 pipes (su3_fx.cuh); the direction mu is a run-time
// argument, so that one copy of its code serves the four directions.
//
// The same update in FP64 arithmetic kept the FP64 pipe (two lanes per SM) busy
// for 93 % of 13.2 ms per 32^4 sweep.  With the matrix products of the staple,
// the rotations and the reunitarisation on the integer multiplier and FP32 (1.76
// SM cycles per multiply-add and warp instead of 16) a sweep took 5.15 ms; with
// the scalars of the proposals there too (su3_fx_kp.cuh) and the subgroups in
// one loop (instruction fetch had become the largest stall: 2.4 of 6.6 cycles
// per instruction) 3.90 ms.  Now 20,000 instructions per warp at 0.51 issued
// per cycle and scheduler; waits for instructions are still the first stall.
#include "su3_kernels.h"

#include "su3_device.cuh"
#include "su3_reduce.cuh"
#include "su3_sweepq.cuh"
#include "su3_update.cuh"

using namespace su3dev;

// Registers per thread.  GB300, 32^4, ms per sweep: 128 registers 4.52, 144: 4.44,
// 168: 4.18, 200: 4.61.  168 is the most that keeps 12 warps on an SM; blocks of
// 256 threads stay legal.
#ifndef SU3_F64_REGS
#define SU3_F64_REGS 168
#endif
#define SU3_F64_BOUNDS __maxnreg__(SU3_F64_REGS)

namespace {

__device__ __forceinline__ UpdateConsts update_consts(const HalfSweepArgs& a) {
  return UpdateConsts{a.three_over_beta_f64, a.three_over_beta, a.max_tries, sweep_far(a.sweep)};
}

// stats != 0: add the acceptance counts (not in measuring phases).
template <bool REPEAT, bool MEAS>
__global__ void SU3_F64_BOUNDS k_half_sweep_f64(HalfSweepArgs args, int mu, int stats) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  UpdateCount c{0, 0};
  double m = 0.0;
  if (h < args.geom.Vh)
    c = update_link_f64<false, REPEAT, MEAS>(args.geom, (double2*)args.links, h, args.parity, mu, *args.sweep, args.key,
                                             update_consts(args), &m);
  if (!MEAS && stats) count_stats<true>(c, args.stats);
  if (MEAS) block_partial(m, args.meas);
}

// The FP64 sweep as four persistent launches, one per direction mu with its
// even and odd half-sweeps, chained by programmatic dependent launch
// (su3_sweepq.cuh): a block takes a tile of `threads` sites of one parity in
// one x3 layer of the lattice and waits only for the layers of the previous
// half-sweep that its staples read, so one half-sweep's last wave overlaps
// the next one's first and only one launch tail per sweep remains.  The
// links change while the launch runs, so they are read through L2 (CG); the
// update is that of k_half_sweep_f64, bit for bit.
template <bool REPEAT>
__global__ void SU3_F64_BOUNDS
    k_sweep_f64(HalfSweepArgs args, SweepQueue qa, int tiles_per_layer, int layers, int stats, int mu) {
  __shared__ SweepItem s_item;
  signal_dependents();
  take_sweep_item<2>(qa, 2 * mu, mu, tiles_per_layer, layers, &s_item);
  __syncthreads();
  const SweepItem it = s_item;
  if (it.phase < 0) return;
  const int h = it.tile * (int)blockDim.x + (int)threadIdx.x;  // layers are whole tiles: always a site of the lattice
  const UpdateCount c = update_link_f64<true, REPEAT>(args.geom, (double2*)args.links, h, it.phase & 1, mu, *args.sweep,
                                                      args.key, update_consts(args));
  if (stats) count_stats<true>(c, args.stats);
  report_sweep_item(qa, layers, it);
}

// One FP64 half-sweep (phase 2 mu + parity) of the chained sweep: one block
// per tile of sites of one x3 layer, the tile from the block's index
// (su3_sweepq.cuh), waiting only for the layers of the previous launch's
// half-sweep that its staples read.
template <bool REPEAT>
__global__ void SU3_F64_BOUNDS
    k_half_sweep_f64_chain(HalfSweepArgs args, SweepQueue qa, int tiles_per_layer, int layers, int stats, int mu,
                           int parity) {
  __shared__ SweepItem s_item;
  signal_dependents();
  own_sweep_item(qa, 2 * mu + parity, tiles_per_layer, layers, &s_item);
  __syncthreads();
  const SweepItem it = s_item;
  if (it.phase < 0) return;
  const int h = it.tile * (int)blockDim.x + (int)threadIdx.x;  // layers are whole tiles: always a site of the lattice
  const UpdateCount c = update_link_f64<true, REPEAT>(args.geom, (double2*)args.links, h, parity, mu, *args.sweep,
                                                      args.key, update_consts(args));
  if (stats) count_stats<true>(c, args.stats);
  report_sweep_item(qa, layers, it);
}

// A small lattice's half-sweep has too few links to fill the GPU, and each
// link's update is a long dependent chain: the time is its latency.  Here four
// lanes share one link: lanes 0, 1, 2 compute rows 0,1 of the two staple paths
// of the first, second and third direction nu != mu at the same time, lane 0
// gathers them and adds them up in the single-thread order (forward then
// backward path, nu ascending, row 2 formed in the accumulation), so the
// staple, and everything after it, is bit for bit that of k_half_sweep_f64.
// Lane 3 only idles.
__device__ __forceinline__ fx_rows01 shfl_rows01(const fx_rows01& m, int src) {
  fx_rows01 r;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const fx &a = m.e[i][k].re, &b = m.e[i][k].im;
      r.e[i][k].re = fx_make(__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src));
      r.e[i][k].im = fx_make(__shfl_sync(0xffffffffu, b.h, src), __shfl_sync(0xffffffffu, b.l, src));
    }
  return r;
}

__global__ void __launch_bounds__(kMaxSweepThreads) k_half_sweep_f64_split(HalfSweepArgs args, int mu, int stats) {
  const Geometry& g = args.geom;
  const int p = args.parity;
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  const int link = gid >> 2, part = gid & 3;
  const bool active = link < g.Vh;
  const int h = active ? link : 0;  // a group past the end works on site 0 and discards it (shuffles stay converged)
  double2* U = (double2*)args.links;
  const UpdateConsts uc = update_consts(args);
  UpdateCount c{0, 0};
  if (*(volatile const int*)uc.far) {  // links far from SU(3): one lane per link
    if (part == 0 && active) c = update_link_f64_far<false>(g, U, h, p, mu, *args.sweep, args.key, uc, nullptr);
  } else {
    const Site st = site_of(g, h, p);
    fx_rows01 F{}, B{};
    if (part < 3) {
      const int nu = part < mu ? part : part + 1;
      const int h_mnu = nb_half_rt(g, st, nu, -1);
      F = staple_path_fx<false>(U, g.Vh, p, mu, nu, false, nb_half_rt(g, st, mu, +1), nb_half_rt(g, st, nu, +1), h);
      B = staple_path_fx<false>(U, g.Vh, p, mu, nu, true, nb_half2_rt(g, st, mu, nu), h_mnu, h_mnu);
    }
    const int lane0 = (threadIdx.x & 31) & ~3;
    fx_staple A;
    fx_staple_zero(A);
    fx_staple_add(A, F);
    fx_staple_add(A, B);
#pragma unroll 1
    for (int k = 1; k < 3; ++k) {
      fx_staple_add(A, shfl_rows01(F, lane0 + k));
      fx_staple_add(A, shfl_rows01(B, lane0 + k));
    }
    if (part == 0 && active) {
      const fx_mat m = fx_staple_mat(A);
      c = heatbath_fx<false, false, false>(g, U, h, p, mu, *args.sweep, (uint32_t)canon(g, st), args.key, uc, m, m,
                                           nullptr);
    }
  }
  if (stats) count_stats<true>(c, args.stats);
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
// Chained half-sweeps or persistent launches of a sweep: launch 0 waits for
// the stream, the others are programmatic dependent launches (su3_sweepq.cuh).
template <bool REPEAT>
cudaError_t launch_sweep_f64(const HalfSweepArgs& a, const SweepQueue& q, int tpl, int layers, bool stats, int threads,
                             bool chained, cudaStream_t s) {
  const int st = stats ? 1 : 0;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(chained ? tpl * layers : 2 * tpl * layers);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cfg.attrs = attr;
  for (int mu = 0; mu < 4; ++mu)
    for (int p = 0; p < (chained ? 2 : 1); ++p) {
      cfg.numAttrs = mu == 0 && p == 0 ? 0 : 1;
      const cudaError_t e = chained
                                ? cudaLaunchKernelEx(&cfg, k_half_sweep_f64_chain<REPEAT>, a, q, tpl, layers, st, mu, p)
                                : cudaLaunchKernelEx(&cfg, k_sweep_f64<REPEAT>, a, q, tpl, layers, st, mu);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace

cudaError_t su3k_launch_half_sweep_f64(const HalfSweepArgs& a, int mu, bool stats, int threads, cudaStream_t s) {
  const int blocks = (a.geom.Vh + threads - 1) / threads;
  const bool repeat = a.max_tries > 1;
  const int st = stats ? 1 : 0;
  if (mu > 0 && a.meas) {  // fused plaquette (statistics are not counted in these phases)
    if (repeat)
      k_half_sweep_f64<true, true><<<blocks, threads, 0, s>>>(a, mu, 0);
    else
      k_half_sweep_f64<false, true><<<blocks, threads, 0, s>>>(a, mu, 0);
  } else if (a.split && !repeat) {
    k_half_sweep_f64_split<<<(4 * a.geom.Vh + threads - 1) / threads, threads, 0, s>>>(a, mu, st);
  } else if (repeat) {
    k_half_sweep_f64<true, false><<<blocks, threads, 0, s>>>(a, mu, st);
  } else {
    k_half_sweep_f64<false, false><<<blocks, threads, 0, s>>>(a, mu, st);
  }
  return cudaGetLastError();
}

int su3k_f64_sweep_layers(const Geometry& g, int threads, int* tiles_per_layer) {
  const long long per_layer = (long long)g.hL0 * g.L1 * g.L2;  // sites of one parity in one x3 layer
  if (threads <= 0 || threads > kMaxSweepThreads || per_layer % threads != 0 || g.L3 < 4) return 0;
  *tiles_per_layer = (int)(per_layer / threads);
  return g.L3;
}

cudaError_t su3k_launch_sweep_f64(const HalfSweepArgs& a, const SweepQueue& q, bool stats, int threads, bool chained,
                                  cudaStream_t s) {
  int tpl = 0;
  const int layers = su3k_f64_sweep_layers(a.geom, threads, &tpl);
  if (layers == 0 || a.meas || a.split) return cudaErrorInvalidValue;
  return a.max_tries > 1 ? launch_sweep_f64<true>(a, q, tpl, layers, stats, threads, chained, s)
                         : launch_sweep_f64<false>(a, q, tpl, layers, stats, threads, chained, s);
}

SU3_BOUNDS_STATUS_FN(su3k_bounds_status_f64)
