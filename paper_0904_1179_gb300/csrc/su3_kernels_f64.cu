// su3_kernels_f64.cu -- the half-sweeps of the FP64 store (see su3_kernels.cu):
// one thread per link, or four or eight lanes per link on small lattices.  The update
// runs on the integer and FP32 pipes (su3_fx.cuh); the direction mu is a run-time
// argument, so that one copy of its code serves the four directions.
//
// The same update in FP64 arithmetic kept the FP64 pipe (two lanes per SM) busy
// for 93 % of 13.2 ms per 32^4 sweep.  What changed it, ms per sweep: the matrix
// products of the staple, the rotations and the reunitarisation on the integer
// multiplier and FP32 (1.76 SM cycles per multiply-add and warp instead of 16)
// 5.15; the scalars of the proposals there too (su3_fx_kp.cuh) and the subgroups
// in one loop (instruction fetch had become the largest stall) 3.90; the staple's
// links copied ahead into shared memory and no spills 3.35; neighbour steps
// looked up and row pairs on the paired FMA 3.20.  Now 16,700 instructions per
// warp at 0.56 issued per cycle and scheduler; what holds the rest are
// fixed-latency dependencies (1.1 of 5.2 cycles per instruction), the shared
// integer pipe (0.7), dispatch (0.6) and instruction fetch (0.5) at three warps
// per scheduler, which 168 registers allow.
// DRAM moves at a quarter of its rate.
#include "su3_kernels.h"

#include "su3_device.cuh"
#include "su3_plaquette.cuh"
#include "su3_reduce.cuh"
#include "su3_sweepq.cuh"
#include "su3_update.cuh"

using namespace su3dev;

// Registers per thread.  GB300, ms per sweep of 32^4 / 24^4 in eight launches: 128
// registers 3.61 / 1.267, 136: 3.32 / 1.149, 144: 3.45 / 1.171, 168: 3.20 / 1.120.
// 168 is the most that keeps 12 warps on an SM; blocks of 256 threads stay legal.
// Spilled at 168, bytes stored: nothing in the one-hit forms of one, four and eight lanes and
// of the per-direction launches, 16 in the chained one; 40, 52 and 36 in the repeat forms of
// one lane, per direction and chained; 156 and 224 in the measuring forms.
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
    c = update_link_f64<REPEAT, MEAS>(args.geom, (double2*)args.links, h, args.parity, mu, *args.sweep, args.key,
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
// links change while the launch runs: the waiting block's acquire drops the SM's
// L1 lines before its cp.async copies go through L1 (copies past L1, .cg, took
// 1.50 ms per 24^4 sweep instead of 1.05); the update is that of k_half_sweep_f64,
// bit for bit.
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
  const UpdateCount c = update_link_f64<REPEAT>(args.geom, (double2*)args.links, h, it.phase & 1, mu, *args.sweep,
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
  const UpdateCount c = update_link_f64<REPEAT>(args.geom, (double2*)args.links, h, parity, mu, *args.sweep,
                                                      args.key, update_consts(args));
  if (stats) count_stats<true>(c, args.stats);
  report_sweep_item(qa, layers, it);
}

// A small lattice's half-sweep: LPL lanes per link (update_link_f64_lanes).
// Launched as a programmatic dependent of the half-sweep before it, a block
// draws its random numbers while that one drains.
template <int LPL, bool REPEAT>
__global__ void SU3_F64_BOUNDS k_half_sweep_f64_lanes(HalfSweepArgs args, int mu, int stats) {
  signal_dependents();
  const int gid = blockIdx.x * blockDim.x + threadIdx.x;
  const int link = gid / LPL;
  const bool active = link < args.geom.Vh;  // a group past the end works on site 0 (shuffles stay converged)
  const UpdateCount c = update_link_f64_lanes<LPL, REPEAT>(args.geom, (double2*)args.links, active ? link : 0,
                                                                 args.parity, mu, args.sweep, args.key,
                                                                 update_consts(args), active);
  if (stats) count_stats<true>(c, args.stats);
}

__global__ void __launch_bounds__(kPlaqFxThreads) k_plaquette_fx(PlaqArgs args, const int* far) {
  plaq_block_fx(args.geom, args.links, far, (int)blockIdx.x, args.partials + blockIdx.x);
}

__global__ void __launch_bounds__(1024) k_plaquette_fx_final(const double* partials, int n, double scale, double* out) {
  sum_partials(partials, n, scale, out);
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
  cfg.dynamicSmemBytes = (size_t)threads * kFxThreadBytes;
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
  const size_t smem = (size_t)threads * kFxThreadBytes;
  if (mu > 0 && a.meas) {  // fused plaquette (statistics are not counted in these phases)
    if (repeat)
      k_half_sweep_f64<true, true><<<blocks, threads, smem, s>>>(a, mu, 0);
    else
      k_half_sweep_f64<false, true><<<blocks, threads, smem, s>>>(a, mu, 0);
  } else if (a.lanes > 1) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(((long long)a.lanes * a.geom.Vh + threads - 1) / threads));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = a.chained ? 1 : 0;
    if (a.lanes == 8)
      return repeat ? cudaLaunchKernelEx(&cfg, k_half_sweep_f64_lanes<8, true>, a, mu, st)
                    : cudaLaunchKernelEx(&cfg, k_half_sweep_f64_lanes<8, false>, a, mu, st);
    return repeat ? cudaLaunchKernelEx(&cfg, k_half_sweep_f64_lanes<4, true>, a, mu, st)
                  : cudaLaunchKernelEx(&cfg, k_half_sweep_f64_lanes<4, false>, a, mu, st);
  } else if (repeat) {
    k_half_sweep_f64<true, false><<<blocks, threads, smem, s>>>(a, mu, st);
  } else {
    k_half_sweep_f64<false, false><<<blocks, threads, smem, s>>>(a, mu, st);
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

int su3k_plaquette_f64_blocks(const Geometry& g) { return plaq_fx_blocks(g); }

cudaError_t su3k_launch_plaquette_f64(const PlaqArgs& a, const int* far, double* out, cudaStream_t s) {
  const int blocks = plaq_fx_blocks(a.geom);
  k_plaquette_fx<<<blocks, kPlaqFxThreads, 0, s>>>(a, far);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_plaquette_fx_final<<<1, 1024, 0, s>>>(a.partials, blocks, 1.0 / (3.0 * 6.0 * 2.0 * (double)a.geom.Vh), out);
  return cudaGetLastError();
}

// The ring takes up to 108 KiB of dynamic shared memory (256 threads of 432 B).
cudaError_t su3k_prepare_f64() {
  const void* const k[] = {(const void*)k_half_sweep_f64<false, false>, (const void*)k_half_sweep_f64<true, false>,
                           (const void*)k_half_sweep_f64<false, true>,  (const void*)k_half_sweep_f64<true, true>,
                           (const void*)k_sweep_f64<false>,             (const void*)k_sweep_f64<true>,
                           (const void*)k_half_sweep_f64_chain<false>,  (const void*)k_half_sweep_f64_chain<true>,
                           (const void*)k_half_sweep_f64_lanes<4, false>, (const void*)k_half_sweep_f64_lanes<4, true>,
                           (const void*)k_half_sweep_f64_lanes<8, false>, (const void*)k_half_sweep_f64_lanes<8, true>};
  for (const void* f : k) {
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSweepThreads * kFxThreadBytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

SU3_BOUNDS_STATUS_FN(su3k_bounds_status_f64)
