// su3_api.cu -- host runtime of libsu3 and its C ABI (include/su3.h).
//
// A handle owns the device link store, the sweep counter (the RNG position),
// the plaquette scratch, the acceptance counters, a staging buffer for layout
// conversion and the instantiated CUDA graphs of one sweep.  The timing
// programs of Berg & Wu (Sec. 2) run `nequi` sweeps with nothing else in the
// loop; su3_sweep replays a graph of the eight half-sweeps for each of them.
#include <cuda.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>

#include "su3_runtime.h"

namespace {

thread_local char g_err[512] = "";

}  // namespace

int su3_fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return code;
}

int su3_cuda_fail(cudaError_t e, const char* what) {
  if (e == cudaErrorMemoryAllocation) return su3_fail(SU3_ENOMEM, "%s: %s", what, cudaGetErrorString(e));
  return su3_fail(SU3_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

int su3_sync(su3_lattice* h, const char* what) {
  if (h->d_pstatus)  // read with the stream's other work: one wait
    SU3_CUDA(cudaMemcpyAsync(h->h_pstatus, h->d_pstatus, sizeof(int), cudaMemcpyDeviceToHost, h->stream), what);
  SU3_CUDA(cudaStreamSynchronize(h->stream), what);
  SU3_CUDA(cudaGetLastError(), what);
  if (h->d_pstatus) {
    if (*h->h_pstatus != 0) {
      // (on the handle's stream: the next sweep reads both words)
      SU3_CUDA(cudaMemsetAsync(h->d_pstatus, 0, sizeof(int), h->stream), what);
      // links that the sweep did not reach keep whatever they held
      h->far_possible = h->precision == SU3_FP64;
      h->half_sweeps = 0;
      SU3_CUDA(cudaMemsetAsync(su3dev::sweep_far(h->d_sweep), 1, sizeof(int), h->stream), what);
      return su3_fail(SU3_ETIMEOUT,
                      "%s: a sweep gave up waiting for tiles of the previous half-sweep (bounded wait of %.3f s); "
                      "the configuration is incomplete",
                      what, (double)h->pq_wait_ns * 1e-9);
    }
  }
  return SU3_OK;
}

namespace {

int fail(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  return su3_fail(code, "%s", buf);
}

int cuda_fail(cudaError_t e, const char* what) { return su3_cuda_fail(e, what); }

constexpr int kDefaultThreads = kSu3DefaultThreads;

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return sms;
}

// Whether a lattice counts as small: its half-sweeps are bound by the latency of
// one update and run several lanes per link, and the persistent and chained
// schedules do not apply.  FP64: at most four warps per SM at four lanes per
// link.  FP32 (k_half_sweep_f32_split): at most eight (8^4 1.35x, 10^4 1.27x;
// 12^4 would lose: 0.92x).
bool use_split(int Vh, int precision) {
  const int sms = sm_count();
  const long long warps_per_sm = precision == SU3_FP64 ? 4 : 8;
  return sms > 0 && 4LL * Vh <= 32LL * warps_per_sm * sms;
}

// Whether the one-hit half-sweeps of a site-paired FP32 store run one thread per
// link (k_half_sweep_f32_single) instead of one per pair: up to 2.5 warps of
// links per scheduler, where twice the threads, each half as long, still fill
// the GPU less than once.  GB300, ms per sweep, per pair / per link (mixed; EFT):
// 12^4 (0.5 warps) 0.078 / 0.056; 0.066 / 0.051, 16^4 (1.7) 0.078 / 0.074; 0.068 /
// 0.064, 16^3 x 20 (2.1) 0.105 / 0.095; 0.084 / 0.080, 20^3 x 16 (3.3) 0.107 /
// 0.121; 0.088 / 0.105, 24^3 x 16 (5.7) 0.135 / 0.173; 0.119 / 0.146.
bool pairs_single(int Vh) {
  const int sms = sm_count();
  return sms > 0 && 2LL * Vh <= 5LL * 32 * 4 * sms;
}

// Lanes per link of an FP64 half-sweep launched by itself
// (k_half_sweep_f64_lanes), by the warps per SM they make.  GB300, ms per sweep
// with 1 / 4 / 8 lanes: 4^4 0.191 / 0.088 / 0.074, 6^4 0.191 / 0.090 / 0.076, 8^4
// (3.4 warps per SM at eight lanes) 0.195 / 0.092 / 0.086, 8^3 x 16 (6.7 at eight,
// 3.4 at four) 0.199 / 0.102 / 0.109, 10^4 0.201 / 0.123 / 0.135, 12^4 (8.5 at four)
// 0.201 / 0.162 / 0.214, 14^4 (15.8) 0.201 / 0.228 / 0.328, 16^4 0.266 / 0.364 /
// 0.570: eight lanes up to four warps per SM (one per scheduler), four up to ten.
int f64_lanes_auto(int Vh) {
  const int sms = sm_count();
  if (sms <= 0) return 1;
  if (8LL * Vh <= 4 * 32LL * sms) return 8;
  return 4LL * Vh <= 10 * 32LL * sms ? 4 : 1;
}

// Default block size for a half-sweep of Vh links: 128 threads, fewer (down
// to one warp) when that would leave SMs idle, so that a small lattice's
// links spread over as many SMs as there are warps (each link's update is a
// long serial chain).
int default_threads(int Vh) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      sms <= 0) {
    cudaGetLastError();
    return kDefaultThreads;
  }
  int t = kDefaultThreads;
  while (t > 32 && (Vh + t - 1) / t < sms) t /= 2;
  return t;
}

}  // namespace

namespace {

void drop_graphs(su3_lattice* h) {
  for (auto& g : h->graph)
    if (g) {
      cudaGraphExecDestroy(g);
      g = nullptr;
    }
  if (h->graph_meas) {
    cudaGraphExecDestroy(h->graph_meas);
    h->graph_meas = nullptr;
  }
}

void release(su3_lattice* h) {
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream);
  drop_graphs(h);
  cudaFree(h->d_pq);
  cudaFree(h->d_pstatus);
  cudaFreeHost(h->h_pstatus);
  if (h->batch) su3_batch_release(h->batch);
  if (h->decomp) su3_decomp_release(h->decomp);
  cudaFree(h->links);
  cudaFree(h->d_sweep);
  cudaFree(h->d_stats);
  cudaFree(h->d_partials);
  cudaFree(h->d_stage);
  cudaFree(h->d_stage2);
  cudaFree(h->d_meas_parts);
  cudaFreeHost(h->h_meas);
  for (int b = 0; b < 2; ++b) {
    if (h->ev_copied[b]) cudaEventDestroy(h->ev_copied[b]);
    if (h->ev_conv[b]) cudaEventDestroy(h->ev_conv[b]);
  }
  if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
  cudaFreeHost(h->h_plaq);
  cudaFreeHost(h->h_stats);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
}

// Whether the FP64 half-sweeps with several lanes per link are programmatic
// dependents of each other: their draws then run while the half-sweep before
// drains, but a programmatic launch costs about 1 us more than a plain one, and
// the early warps take issue slots from the last.  GB300, ms per sweep, plain /
// programmatic: 4^4 (0.2 warps per SM) 0.084 / 0.076, 6^4 (1.1) 0.088 / 0.080,
// 8^4 (3.4) 0.090 / 0.095, 8^3 x 16 (3.4 at four lanes) 0.111 / 0.118, 10^4 (4.1)
// 0.131 / 0.140, 12^4 (8.5) 0.178 / 0.168.  (Without draws to overlap it only
// costs: the FP32 half-sweeps of 8^4 to 24^3 x 16 took 8 to 25 % longer.)
bool f64_lanes_chained(const su3_lattice* h) {
  const int sms = sm_count(), lanes = su3_f64_lanes(h);
  const long long threads = (long long)lanes * h->geom.Vh;
  return sms > 0 && lanes > 1 && (threads <= 2 * 32LL * sms || threads >= 8 * 32LL * sms);
}

HalfSweepArgs half_sweep_args(const su3_lattice* h, int parity, int threads) {
  HalfSweepArgs a{};
  a.meas = nullptr;
  a.split = h->split;
  a.lanes = h->precision == SU3_FP64 ? su3_f64_lanes(h) : 1;
  a.pairs = h->pairs;
  a.single = h->pairs && pairs_single(h->geom.Vh);
  a.pgeom = h->pgeom;
  a.tile2 = h->pairs ? su3k_pair_tile2(h->pgeom, threads) : 0;
  a.geom = h->geom;
  a.key = su3dev::philox_round_keys(h->key);
  a.parity = parity;
  a.beta = h->beta;
  a.three_over_beta = (float)(3.0 / h->beta);
  a.three_over_beta_f64 = 3.0 / h->beta;
  a.max_tries = h->max_tries;
  a.sweep = h->d_sweep;
  a.links = h->links;
  a.stats = h->d_stats;
  return a;
}

// Whether the sweep can run as persistent launches: the site-paired FP32
// store with one lane per link and a pair lattice whose x3 layers are whole
// tiles (one launch per sweep or one per direction, su3k_launch_sweep_pair);
// or the FP64 store with one lane per link and x3 layers of whole tiles (one
// launch per direction, su3k_launch_sweep_f64).
bool pair_persistent_applies(const su3_lattice* h, int threads) {
  int tpl = 0;
  return h->pairs && !h->split && su3k_pair_sweep_layers(h->pgeom, threads, &tpl) > 0;
}
bool f64_persistent_applies(const su3_lattice* h, int threads) {
  int tpl = 0;
  return h->precision == SU3_FP64 && !h->split && su3k_f64_sweep_layers(h->geom, threads, &tpl) > 0;
}

bool persistent_applies(const su3_lattice* h, int threads) {
  return pair_persistent_applies(h, threads) || f64_persistent_applies(h, threads);
}

// Waves of the GPU in one half-sweep: site pairs at about 512 threads per SM
// (128 registers), FP64 links at 384 (3 warps of 168 registers per
// scheduler).
double half_sweep_waves(const su3_lattice* h) {
  const int sms = sm_count();
  if (sms <= 0) return 1e9;
  return h->pairs ? (double)h->pgeom.Vh / (512.0 * sms) : (double)h->geom.Vh / (384.0 * sms);
}

// SU3_SCHED_AUTO by the number of waves of a half-sweep, after measurements
// on GB300 against eight launches.  Site-paired FP32 (mixed / EFT), the eight
// chained half-sweep launches: 24^4 (1.1 waves) +15 / +17 %, 32^4 (3.4 waves)
// +10 / +6 %, 32^3 x 64 (6.7 waves) +3.4 / +0.9 %, 40^4 (8.2 waves) +0.8 /
// +0.1 %, 48^4 (17 waves) -2.4 / -2.4 %: chained below 10 waves.  FP64, one
// launch per direction: 24^4 (2.8 waves) +8 %, 32^4 (9 waves) +1.6 %, 40^4 -0.2 %,
// 48^4 -1.3 %: per direction below 5 waves (the documented
// default of 32^4 is eight launches).  Under one wave a whole half-sweep is
// in flight at once and the tiles of the next one wait on it (FP32 per direction:
// 24^3 x 16, 0.7 waves, -38 %; 16^4, 0.2 waves, -62 %; FP64 16^4, 0.6 waves, -28 %):
// eight launches.
int auto_schedule(const su3_lattice* h) {
  const double w = half_sweep_waves(h);
  if (h->pairs) return w >= 1.0 && w < 10.0 ? SU3_SCHED_CHAINED : SU3_SCHED_PHASES;
  return w >= 1.0 && w < 5.0 ? SU3_SCHED_PER_DIRECTION : SU3_SCHED_PHASES;
}

// Whether a schedule other than eight independent launches applies to h.
bool schedule_applies(const su3_lattice* h, int schedule) {
  switch (schedule) {
    case SU3_SCHED_PERSISTENT: return pair_persistent_applies(h, h->threads);
    case SU3_SCHED_CHAINED:
    case SU3_SCHED_PER_DIRECTION: return persistent_applies(h, h->threads);
    default: return true;
  }
}

// Threads per tile of the automatic schedule, 0 where that is eight launches:
// the default block size or, unless the caller set the block size, the largest
// smaller one that an x3 layer is a whole number of.  The schedule gains most
// just above one wave, and blocks of one or two warps cost up to 3 %, so the FP32
// store takes them below three waves only.  GB300, ms per sweep, eight launches of
// 128 / smaller tiles: FP64 20^4 (1.4 waves, 32 threads) 0.598 / 0.529, 20^2 x 24 x 20
// (1.6, 64) 0.645 / 0.605, 26 x 24^3 (3.1, 64) 1.196 / 1.101; FP32 mixed (EFT) 26 x
// 24^3 (1.2, 64) 0.211 / 0.202 (0.187 / 0.175), 28^4 (2.0, 32) 0.322 / 0.283 (0.294 /
// 0.272), 36^4 (5.4, 32) 0.763 / 0.756 (0.707 / 0.716).
int schedule_tile(const su3_lattice* h) {
  if (auto_schedule(h) == SU3_SCHED_PHASES) return 0;
  if (persistent_applies(h, h->threads)) return h->threads;
  if (h->threads_set || (h->pairs && half_sweep_waves(h) >= 3.0)) return 0;
  for (int t = h->threads / 2; t >= 32; t /= 2)
    if (persistent_applies(h, t)) return t;
  return 0;
}

// The schedule the next sweep runs with (measuring sweeps: always eight
// launches).
int effective_schedule(const su3_lattice* h, bool measured = false) {
  if (measured) return SU3_SCHED_PHASES;
  if (h->schedule == SU3_SCHED_AUTO) return schedule_tile(h) ? auto_schedule(h) : SU3_SCHED_PHASES;
  return schedule_applies(h, h->schedule) ? h->schedule : SU3_SCHED_PHASES;
}

// Threads per block of the next sweep's launches: h->threads, or the automatic
// schedule's tile, or, for an FP32 half-sweep of less than 0.8 waves (of 512
// threads per SM) whose block size the caller left alone, one warp: blocks of 128
// then leave some SMs with twice the warps of others.  GB300, ms per sweep, 128 / 32
// threads, mixed (EFT): 18 x 10 x 14 x 22 (0.36 waves) 0.060 / 0.056 (0.050 / 0.050),
// 16^4 0.074 / 0.070 (0.063 / 0.060), 16^3 x 20 0.097 / 0.084 (0.080 / 0.076), 20 x 18^2
// x 20 (0.4) 0.151 / 0.103 (0.128 / 0.087), 20^4 (0.5) 0.153 / 0.128 (0.132 / 0.115), 24^3 x
// 16 (0.71) 0.138 / 0.138 (0.119 / 0.119), 22^3 x 24 (0.75) 0.197 / 0.174 (0.179 / 0.154),
// 24^3 x 20 (0.89) 0.172 / 0.176 (0.154 / 0.154).  FP64 blocks of one warp fill the
// schedulers unevenly (18^4 0.377 / 0.439).  Measuring sweeps keep h->threads: the
// order of their plaquette sums follows the blocks.
int launch_threads(const su3_lattice* h, bool measured = false) {
  if (h->threads_set || measured) return h->threads;
  if (effective_schedule(h) != SU3_SCHED_PHASES) return h->schedule == SU3_SCHED_AUTO ? schedule_tile(h) : h->threads;
  const int sms = sm_count();
  const long long n = h->pairs && !pairs_single(h->geom.Vh) ? h->pgeom.Vh : h->geom.Vh;
  return h->precision != SU3_FP64 && !h->split && sms > 0 && 5 * n < 4 * 512LL * sms ? 32 : h->threads;
}

bool use_persistent(const su3_lattice* h, bool measured = false) {
  return effective_schedule(h, measured) != SU3_SCHED_PHASES;
}

// Counters and status word of the persistent sweep (allocated on first use,
// outside any stream capture).
int ensure_pair_queue(su3_lattice* h) {
  if (h->d_pq) return SU3_OK;
  const int words = su3k_sweep_words(h->pairs ? h->pgeom.L3 : h->geom.L3);
  cudaError_t e;
  if ((e = cudaMalloc(&h->d_pq, (size_t)words * sizeof(unsigned int))) != cudaSuccess ||
      (e = cudaMalloc(&h->d_pstatus, sizeof(int))) != cudaSuccess ||
      (e = cudaMallocHost(&h->h_pstatus, sizeof(int))) != cudaSuccess ||
      (e = cudaMemsetAsync(h->d_pstatus, 0, sizeof(int), h->stream)) != cudaSuccess) {
    cudaFree(h->d_pq);
    cudaFree(h->d_pstatus);
    cudaFreeHost(h->h_pstatus);
    h->d_pq = nullptr;
    h->d_pstatus = nullptr;
    h->h_pstatus = nullptr;
    return cuda_fail(e, "persistent sweep counters");
  }
  h->pq_words = words;
  return SU3_OK;
}

// One sweep: mu = 0..3, even then odd sites, then the sweep counter.  With
// `measured`, the odd-site phases of mu = 1, 2, 3 also leave block partials of
// Re Tr(U_new A_<) (A_< = staple terms of nu < mu); together they hold every
// plaquette of the updated configuration once, and a last kernel sums them
// into the ring slot of this sweep.
int enqueue_sweep_body(su3_lattice* h, bool measured) {
  const int threads = launch_threads(h, measured);
  const int blocks = su3k_half_sweep_blocks(half_sweep_args(h, 1, threads), h->precision, threads);
  if (use_persistent(h, measured)) {
    const HalfSweepArgs a = half_sweep_args(h, 0, threads);
    const SweepQueue q{h->d_pq, h->d_pstatus, h->pq_wait_ns, h->pq_withhold};
    SU3_CUDA(cudaMemsetAsync(h->d_pq, 0, (size_t)h->pq_words * sizeof(unsigned int), h->stream),
             "sweep counters reset");
    if (h->precision == SU3_FP64)
      SU3_CUDA(su3k_launch_sweep_f64(a, q, h->stats_on, threads, effective_schedule(h) == SU3_SCHED_CHAINED,
                                     h->stream),
               "persistent sweep launch");
    else
      SU3_CUDA(su3k_launch_sweep_pair(a, q, h->precision == SU3_FP32_EFT, h->stats_on, threads,
                                      effective_schedule(h) == SU3_SCHED_CHAINED        ? SweepForm::kChained
                                      : effective_schedule(h) == SU3_SCHED_PER_DIRECTION ? SweepForm::kPerDirection
                                                                                         : SweepForm::kOneLaunch,
                                      h->stream),
               "persistent sweep launch");
  } else {
    for (int mu = 0; mu < 4; ++mu)
      for (int p = 0; p < 2; ++p) {
        HalfSweepArgs a = half_sweep_args(h, p, threads);
        a.chained = mu + p > 0 && h->precision == SU3_FP64 && f64_lanes_chained(h);
        if (measured && p == 1 && mu >= 1) a.meas = h->d_meas_parts + (size_t)(mu - 1) * blocks;
        SU3_CUDA(su3k_launch_half_sweep(a, mu, h->precision, h->stats_on, threads, h->stream),
                 "half-sweep launch");
      }
  }
  if (measured)
    SU3_CUDA(su3k_launch_meas_final(h->d_meas_parts, 3 * blocks, 1.0 / (6.0 * (double)h->V), h->d_sweep, h->h_meas,
                                    h->meas_cap, h->stream),
             "plaquette reduction launch");
  SU3_CUDA(su3k_launch_increment(h->d_sweep, 1, su3dev::sweep_far(h->d_sweep), 1, h->stream), "sweep counter launch");
  return SU3_OK;
}

int ensure_graph(su3_lattice* h, bool measured = false) {
  cudaGraphExec_t& exec = measured ? h->graph_meas : h->graph[h->stats_on ? 1 : 0];
  if (exec) return SU3_OK;
  if (use_persistent(h, measured)) {
    const int rc = ensure_pair_queue(h);
    if (rc != SU3_OK) return rc;
  }
  cudaGraph_t graph = nullptr;
  SU3_CUDA(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal), "graph capture begin");
  const int rc = enqueue_sweep_body(h, measured);
  const cudaError_t e = cudaStreamEndCapture(h->stream, &graph);
  if (rc != SU3_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(e, "graph capture end");
  const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ei != cudaSuccess) {
    exec = nullptr;
    return cuda_fail(ei, "graph instantiate");
  }
  return SU3_OK;
}

int sync(su3_lattice* h, const char* what) { return su3_sync(h, what); }

// Single-lattice calls reject batch handles and vice versa.
bool is_batch(const su3_lattice* h) { return h && h->batch; }

// After a half-sweep called by itself: once all eight have run since the flags were
// last set or moved (links_set, a timeout, a sweep, this function), every link has been rewritten and the flags move
// on as at the end of a sweep (nothing else would end the FP64 arithmetic of a chain
// driven by half-sweeps).
int note_half_sweep(su3_lattice* h, int mu, int parity) {
  if (!h->far_possible) return SU3_OK;
  h->half_sweeps |= 1u << (2 * mu + parity);
  if (h->half_sweeps != 0xffu) return SU3_OK;
  h->half_sweeps = 0;
  SU3_CUDA(su3k_launch_increment(h->d_sweep, 0, su3dev::sweep_far(h->d_sweep), 1, h->stream), "su3_half_sweep");
  return SU3_OK;
}

}  // namespace

void su3_release_handle(su3_lattice* h) { release(h); }

int su3_f64_lanes(const su3_lattice* h) { return h->lanes ? h->lanes : f64_lanes_auto(h->geom.Vh); }

int su3_internal_fail(int code, const char* msg) { return su3_fail(code, "%s", msg); }

namespace {

// Second staging buffer, copy stream and events of the transfer pipeline,
// created on first use.
int ensure_transfer(su3_lattice* h, const char* what) {
  if (h->copy_stream) return SU3_OK;
  const long long chunk = h->V < kChunkSites ? h->V : kChunkSites;
  SU3_CUDA(cudaMalloc(&h->d_stage2, (size_t)chunk * 72 * sizeof(double)), what);
  for (int b = 0; b < 2; ++b) {
    SU3_CUDA(cudaEventCreateWithFlags(&h->ev_copied[b], cudaEventDisableTiming), what);
    SU3_CUDA(cudaEventCreateWithFlags(&h->ev_conv[b], cudaEventDisableTiming), what);
  }
  SU3_CUDA(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking), what);
  return SU3_OK;
}

}  // namespace

// The GPU's address of a host buffer that a kernel may write, or null: all of it in
// one page-locked allocation or registration (between two lie pages that the GPU may
// not write or that nobody mapped), not registered read-only, on a GPU that shares
// the host's page tables, 16-byte aligned.  (The driver call is resolved through the
// runtime, so that libsu3 does not link the driver library.)
static double* host_direct(su3_lattice* h, double* host, size_t bytes) {
  typedef CUresult (*AttributesFn)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);
  static const AttributesFn attributes = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool found = cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q) ==
                           cudaSuccess &&
                       q == cudaDriverEntryPointSuccess;
    return found ? (AttributesFn)f : (AttributesFn) nullptr;
  }();
  if (h->shared_tables < 0) {  // of the handle's GPU: asked once
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->shared_tables, cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
  }
  unsigned flags = 0;
  if (!attributes || !h->shared_tables || ((uintptr_t)host & 15)) return nullptr;
  if (cudaHostGetFlags(&flags, host) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (flags & cudaHostRegisterReadOnly) return nullptr;
  CUpointer_attribute what[3] = {CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE,
                                 CU_POINTER_ATTRIBUTE_DEVICE_POINTER};
  CUdeviceptr start = 0, device = 0;
  size_t size = 0;
  void* data[3] = {&start, &size, &device};
  if (attributes(3, what, data, (CUdeviceptr)host) != CUDA_SUCCESS || start == 0 || (CUdeviceptr)host < start) return nullptr;
  const size_t before = (size_t)((CUdeviceptr)host - start);
  return before <= size && bytes <= size - before ? (double*)device : nullptr;
}

int su3_transfer(su3_lattice* h, const su3dev::Geometry& g, void* links, bool pairs, int* far, double* host, bool get,
                 const char* what, const int* status, int* status_host) {
  const long long V = 2LL * g.Vh;
  // Page-locked memory: the conversion writes the caller's buffer itself, one launch of any size.  GB300, get through
  // the staging buffer / directly: 4^4 18 / 14 us, 8^4 30 / 26 us (FP32 38 / 28), 16^4 222 / 210 us (FP32 246 / 215),
  // 32^4 3.18 / 3.14 ms, 48^4 15.98 / 15.82 ms (the host link's 193 GB/s: 3.13 and 15.8 ms).
  if (double* direct = get ? host_direct(h, host, (size_t)V * 72 * sizeof(double)) : nullptr) {
    ConvArgs a{g, h->precision, 0, V, direct, links, pairs ? 1 : 0, far};
    a.status = status;
    a.status_host = status_host;
    SU3_CUDA(su3k_launch_conv(a, false, h->stream), what);
    return h->batch ? SU3_OK : su3_sync(h, what);
  }
  if (status)
    SU3_CUDA(cudaMemcpyAsync(status_host, status, sizeof(int), cudaMemcpyDeviceToHost, h->stream), what);
  if (V <= kChunkSites) {
    // one chunk has nothing to overlap: conversion and copy follow each other on
    // the handle's stream, without the events and the second wait (one 8^4 replica of a batch: 52.6 -> 40.0 us)
    ConvArgs a{g, h->precision, 0, V, h->d_stage, links, pairs ? 1 : 0, far};
    a.far_host = h->h_far;
    const size_t bytes = (size_t)V * 72 * sizeof(double);
    if (get) {
      SU3_CUDA(su3k_launch_conv(a, false, h->stream), what);
      SU3_CUDA(cudaMemcpyAsync(host, h->d_stage, bytes, cudaMemcpyDeviceToHost, h->stream), what);
    } else {
      if (far) SU3_CUDA(cudaMemsetAsync(far, 0, 2 * sizeof(int), h->stream), what);
      SU3_CUDA(cudaMemcpyAsync(h->d_stage, host, bytes, cudaMemcpyHostToDevice, h->stream), what);
      SU3_CUDA(su3k_launch_conv(a, true, h->stream), what);
    }
    return h->batch ? SU3_OK : su3_sync(h, what);
  }
  int rc = ensure_transfer(h, what);
  if (rc != SU3_OK) return rc;
  double* stage[2] = {h->d_stage, h->d_stage2};
  // the conversion into the store flags links far from SU(3)
  if (!get && far) SU3_CUDA(cudaMemsetAsync(far, 0, 2 * sizeof(int), h->stream), what);
  int i = 0;
  for (long long s0 = 0; s0 < V; s0 += kChunkSites, ++i) {
    const long long n = (V - s0) < kChunkSites ? (V - s0) : kChunkSites;
    const int b = i & 1;
    cudaStream_t cs = h->copy_stream;
    const size_t bytes = (size_t)n * 72 * sizeof(double);
    ConvArgs a{g, h->precision, s0, n, stage[b], links, pairs ? 1 : 0, far};
    a.far_host = h->h_far;
    if (get) {
      // stage[b] is free once the copy-out of chunk i-2 has finished
      if (i >= 2) SU3_CUDA(cudaStreamWaitEvent(h->stream, h->ev_copied[b], 0), what);
      SU3_CUDA(su3k_launch_conv(a, false, h->stream), what);
      SU3_CUDA(cudaEventRecord(h->ev_conv[b], h->stream), what);
      SU3_CUDA(cudaStreamWaitEvent(cs, h->ev_conv[b], 0), what);
      SU3_CUDA(cudaMemcpyAsync(host + s0 * 72, stage[b], bytes, cudaMemcpyDeviceToHost, cs), what);
      SU3_CUDA(cudaEventRecord(h->ev_copied[b], cs), what);
    } else {
      // stage[b] is free once the conversion of chunk i-2 has read it
      if (i >= 2) SU3_CUDA(cudaStreamWaitEvent(cs, h->ev_conv[b], 0), what);
      SU3_CUDA(cudaMemcpyAsync(stage[b], host + s0 * 72, bytes, cudaMemcpyHostToDevice, cs), what);
      SU3_CUDA(cudaEventRecord(h->ev_copied[b], cs), what);
      SU3_CUDA(cudaStreamWaitEvent(h->stream, h->ev_copied[b], 0), what);
      SU3_CUDA(su3k_launch_conv(a, true, h->stream), what);
      SU3_CUDA(cudaEventRecord(h->ev_conv[b], h->stream), what);
    }
  }
  SU3_CUDA(cudaStreamSynchronize(h->copy_stream), what);
  return h->batch ? SU3_OK : su3_sync(h, what);
}

extern "C" {

const char* su3_last_error(void) { return g_err; }

const char* su3_version(void) { return "libsu3 1.0 (sm_103a)"; }

int su3_create_ex(int L0, int L1, int L2, int L3, double beta, uint64_t seed, int start, int precision, void* cuda_stream,
                  su3_handle* out) {
  if (!out) return fail(SU3_EINVAL, "su3_create: out is NULL");
  *out = nullptr;
  const int L[4] = {L0, L1, L2, L3};
  for (int mu = 0; mu < 4; ++mu)
    if (L[mu] < 2 || (L[mu] & 1))
      return fail(SU3_EINVAL, "su3_create: extent L%d = %d must be even and >= 2", mu, L[mu]);
  const long long V = (long long)L0 * L1 * L2 * L3;
  if (4 * V > 0x7fffffffLL) return fail(SU3_EINVAL, "su3_create: 4*V = %lld exceeds 2^31-1", 4 * V);
  if (!(beta > 0.0) || !std::isfinite(beta)) return fail(SU3_EINVAL, "su3_create: beta must be finite and > 0");
  if (start != SU3_COLD && start != SU3_HOT) return fail(SU3_EINVAL, "su3_create: bad start %d", start);
  if (precision != SU3_FP64 && precision != SU3_FP32_MIXED && precision != SU3_FP32_EFT)
    return fail(SU3_EINVAL, "su3_create: bad precision %d", precision);

  su3_lattice* h = new (std::nothrow) su3_lattice;
  if (!h) return fail(SU3_ENOMEM, "su3_create: host allocation failed");
  for (int mu = 0; mu < 4; ++mu) h->L[mu] = L[mu];
  h->V = V;
  h->beta = beta;
  h->seed = seed;
  h->precision = precision;
  h->geom = su3dev::make_geometry(L0, L1, L2, L3);
  h->pairs = precision != SU3_FP64 && su3_fp32_pairs(L3);
  if (h->pairs) h->pgeom = su3dev::make_geometry(L0, L1, L2, L3 / 2);
  h->key.k0 = (uint32_t)seed;
  h->key.k1 = (uint32_t)(seed >> 32);
  h->threads = default_threads(h->pairs ? h->pgeom.Vh : h->geom.Vh);
  h->split = use_split(h->geom.Vh, precision);
  {
    const cudaError_t ep = precision == SU3_FP64 ? su3k_prepare_f64() : su3k_prepare();
    if (ep != cudaSuccess) {
      delete h;
      return cuda_fail(ep, "su3_create: kernel attributes");
    }
  }

  cudaError_t e;
  if (cuda_stream) {
    h->stream = (cudaStream_t)cuda_stream;
  } else {
    e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      delete h;
      return cuda_fail(e, "su3_create: stream");
    }
    h->own_stream = true;
  }
  // the site-paired FP32 store pads each (mu, parity) array to whole tiles of pairs
  h->link_bytes = h->pairs ? (size_t)8 * 6 * su3dev::pair_padded(V / 4) * sizeof(float4)
                           : (size_t)V * 4 * (precision == SU3_FP64 ? 18 * sizeof(double) : 12 * sizeof(float));
  const int nparts = precision == SU3_FP64 ? su3k_plaquette_f64_blocks(h->geom) : su3k_plaquette_blocks(h->geom);
  const long long chunk = V < kChunkSites ? V : kChunkSites;
  if ((e = cudaMalloc(&h->links, h->link_bytes)) != cudaSuccess ||
      (e = cudaMalloc(&h->d_sweep, sizeof(su3dev::SweepState))) != cudaSuccess ||
      (e = cudaMalloc(&h->d_stats, 2 * sizeof(unsigned long long))) != cudaSuccess ||
      (e = cudaMalloc(&h->d_partials, (size_t)nparts * sizeof(double))) != cudaSuccess ||
      (e = cudaMalloc(&h->d_stage, (size_t)chunk * 4 * 18 * sizeof(double))) != cudaSuccess ||
      (e = cudaMallocHost(&h->h_plaq, sizeof(double))) != cudaSuccess ||
      (e = cudaMallocHost(&h->h_stats, 3 * sizeof(unsigned long long))) != cudaSuccess) {
    const int rc = cuda_fail(e, "su3_create: allocation");
    cudaGetLastError();
    release(h);
    return rc;
  }
  h->h_far = (int*)(h->h_stats + 2);
  *h->h_far = 0;
  int rc = SU3_OK;
  if ((e = cudaMemsetAsync(h->d_sweep, 0, sizeof(su3dev::SweepState), h->stream)) != cudaSuccess ||
      (e = cudaMemsetAsync(h->d_stats, 0, 2 * sizeof(unsigned long long), h->stream)) != cudaSuccess) {
    rc = cuda_fail(e, "su3_create: memset");
  }
  if (rc == SU3_OK) {
    InitArgs ia{h->geom, su3dev::philox_round_keys(h->key), precision, h->links, h->pairs ? 1 : 0};
    e = su3k_launch_init(ia, start == SU3_HOT, h->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "su3_create: start configuration");
  }
  if (rc == SU3_OK) rc = sync(h, "su3_create");
  if (rc != SU3_OK) {
    release(h);
    return rc;
  }
  *out = h;
  return SU3_OK;
}

int su3_create(int L0, int L1, int L2, int L3, double beta, uint64_t seed, int start, su3_handle* out) {
  return su3_create_ex(L0, L1, L2, L3, beta, seed, start, SU3_FP64, nullptr, out);
}

int su3_destroy(su3_handle h) {
  release(h);
  return SU3_OK;
}

int su3_sweep(su3_handle h, int nsweeps) {
  if (!h) return fail(SU3_EINVAL, "su3_sweep: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_sweep: batch handle (use the su3_batch_* calls)");
  if (nsweeps < 0) return fail(SU3_EINVAL, "su3_sweep: nsweeps < 0");
  if (nsweeps == 0) return SU3_OK;
  h->half_sweeps = 0;  // the sweep moves the flags itself
  if (su3_decomp_active(h)) return su3_decomp_sweep(h, nsweeps);
  int rc = ensure_graph(h);
  if (rc != SU3_OK) return rc;
  cudaGraphExec_t exec = h->graph[h->stats_on ? 1 : 0];
  for (int n = 0; n < nsweeps; ++n) SU3_CUDA(cudaGraphLaunch(exec, h->stream), "su3_sweep: graph launch");
  h->sweep_host += (uint64_t)nsweeps;
  return SU3_OK;
}

int su3_sweep_measured(su3_handle h, int nsweeps, double* plaq_out) {
  if (!h) return fail(SU3_EINVAL, "su3_sweep_measured: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_sweep_measured: batch handle (use su3_batch_plaquettes)");
  if (nsweeps < 0 || (nsweeps > 0 && !plaq_out)) return fail(SU3_EINVAL, "su3_sweep_measured: bad nsweeps or NULL out");
  if (h->stats_on) return fail(SU3_EINVAL, "su3_sweep_measured: disable acceptance statistics first");
  if (nsweeps == 0) return SU3_OK;
  h->half_sweeps = 0;
  const bool dec = su3_decomp_active(h);
  const int blocks = dec ? su3_decomp_meas_blocks(h) : su3k_half_sweep_blocks(half_sweep_args(h, 1, h->threads), h->precision, h->threads);
  if (h->meas_blocks != blocks || !h->h_meas) {
    SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_sweep_measured");
    if (h->graph_meas) {
      cudaGraphExecDestroy(h->graph_meas);
      h->graph_meas = nullptr;
    }
    if (h->decomp) su3_decomp_invalidate(h->decomp);  // its graphs hold the old partials buffer
    cudaFree(h->d_meas_parts);
    h->d_meas_parts = nullptr;
    SU3_CUDA(cudaMalloc(&h->d_meas_parts, (size_t)3 * blocks * sizeof(double)), "su3_sweep_measured: partials");
    h->meas_blocks = blocks;
    if (!h->h_meas) {
      h->meas_cap = 4096;
      SU3_CUDA(cudaMallocHost(&h->h_meas, (size_t)h->meas_cap * sizeof(double)), "su3_sweep_measured: ring");
    }
  }
  cudaGraphExec_t exec = nullptr;
  int rc = dec ? su3_decomp_sweep_measured_graph(h, &exec) : ensure_graph(h, true);
  if (rc != SU3_OK) return rc;
  if (!dec) exec = h->graph_meas;
  for (int done = 0; done < nsweeps;) {
    const int n = (nsweeps - done) < h->meas_cap ? (nsweeps - done) : h->meas_cap;
    const uint64_t t0 = h->sweep_host;
    for (int i = 0; i < n; ++i) SU3_CUDA(cudaGraphLaunch(exec, h->stream), "su3_sweep_measured: graph launch");
    h->sweep_host += (uint64_t)n;
    rc = sync(h, "su3_sweep_measured");
    if (rc != SU3_OK) return rc;
    for (int i = 0; i < n; ++i) plaq_out[done + i] = h->h_meas[(t0 + (uint64_t)i) % (uint64_t)h->meas_cap];
    done += n;
  }
  return SU3_OK;
}

int su3_half_sweep(su3_handle h, int mu, int parity) {
  if (!h) return fail(SU3_EINVAL, "su3_half_sweep: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_half_sweep: batch handle (use the su3_batch_* calls)");
  if (mu < 0 || mu > 3 || parity < 0 || parity > 1) return fail(SU3_EINVAL, "su3_half_sweep: bad mu/parity");
  if (su3_decomp_active(h)) {
    const int rc = su3_decomp_half_sweep(h, mu, parity);
    return rc == SU3_OK ? note_half_sweep(h, mu, parity) : rc;
  }
  const int threads = launch_threads(h);
  SU3_CUDA(su3k_launch_half_sweep(half_sweep_args(h, parity, threads), mu, h->precision, h->stats_on, threads, h->stream),
           "su3_half_sweep");
  return note_half_sweep(h, mu, parity);
}

double su3_plaquette(su3_handle h) {
  if (!h || is_batch(h)) {
    fail(SU3_EINVAL, h ? "su3_plaquette: batch handle (use su3_batch_plaquettes)" : "su3_plaquette: NULL handle");
    return NAN;
  }
  if (su3_decomp_sync_global(h) != SU3_OK) return NAN;
  PlaqArgs a{h->geom, h->links, h->d_partials, h->pairs ? 1 : 0};
  cudaError_t e = h->precision == SU3_FP64
                      ? su3k_launch_plaquette_f64(a, su3dev::sweep_far(h->d_sweep), h->h_plaq, h->stream)
                      : su3k_launch_plaquette(a, h->precision, h->h_plaq, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) {
    cuda_fail(e, "su3_plaquette");
    return NAN;
  }
  return *h->h_plaq;
}

int su3_links_get(su3_handle h, double* host, size_t n_doubles) {
  if (!h || !host) return fail(SU3_EINVAL, "su3_links_get: NULL argument");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_links_get: batch handle (use the su3_batch_* calls)");
  if (n_doubles != (size_t)h->V * 72) return fail(SU3_ESIZE, "su3_links_get: n = %zu, expected %lld", n_doubles, h->V * 72);
  const int rc = su3_decomp_sync_global(h);
  if (rc != SU3_OK) return rc;
  return su3_transfer(h, h->geom, h->links, h->pairs, su3dev::sweep_far(h->d_sweep), host, true, "su3_links_get");
}

int su3_links_set(su3_handle h, const double* host, size_t n_doubles) {
  if (!h || !host) return fail(SU3_EINVAL, "su3_links_set: NULL argument");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_links_set: batch handle (use the su3_batch_* calls)");
  if (n_doubles != (size_t)h->V * 72) return fail(SU3_ESIZE, "su3_links_set: n = %zu, expected %lld", n_doubles, h->V * 72);
  *h->h_far = 0;  // (only the conversion below writes it)
  const int rc = su3_transfer(h, h->geom, h->links, h->pairs, su3dev::sweep_far(h->d_sweep),
                              const_cast<double*>(host), false, "su3_links_set");
  h->far_possible = *h->h_far != 0 || (rc != SU3_OK && h->precision == SU3_FP64);
  h->half_sweeps = 0;
  if (rc == SU3_OK) su3_decomp_global_written(h);
  return rc;
}

int su3_sweep_count(su3_handle h, uint64_t* out) {
  if (!h || !out) return fail(SU3_EINVAL, "su3_sweep_count: NULL argument");
  *out = h->sweep_host;
  return SU3_OK;
}

int su3_set_sweep_count(su3_handle h, uint64_t n) {
  if (!h) return fail(SU3_EINVAL, "su3_set_sweep_count: NULL handle");
  SU3_CUDA(su3k_launch_set_counter(h->d_sweep, n, h->stream), "su3_set_sweep_count");
  h->sweep_host = n;
  return SU3_OK;
}

int su3_set_stats(su3_handle h, int enable) {
  if (!h) return fail(SU3_EINVAL, "su3_set_stats: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_set_stats: batch handle (use the su3_batch_* calls)");
  h->stats_on = enable != 0;
  if (h->stats_on)
    SU3_CUDA(cudaMemsetAsync(h->d_stats, 0, 2 * sizeof(unsigned long long), h->stream), "su3_set_stats");
  return SU3_OK;
}

int su3_stats(su3_handle h, uint64_t* accepted, uint64_t* proposed) {
  if (!h || !accepted || !proposed) return fail(SU3_EINVAL, "su3_stats: NULL argument");
  SU3_CUDA(cudaMemcpyAsync(h->h_stats, h->d_stats, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, h->stream),
           "su3_stats");
  const int rc = sync(h, "su3_stats");
  if (rc != SU3_OK) return rc;
  *accepted = h->h_stats[0];
  *proposed = h->h_stats[1];
  return SU3_OK;
}

int su3_info(su3_handle h, int dims[4], double* beta, uint64_t* seed, int* precision) {
  if (!h) return fail(SU3_EINVAL, "su3_info: NULL handle");
  if (dims)
    for (int mu = 0; mu < 4; ++mu) dims[mu] = h->L[mu];
  if (beta) *beta = h->beta;
  if (seed) *seed = h->seed;
  if (precision) *precision = h->precision;
  return SU3_OK;
}

int su3_set_heatbath(su3_handle h, int max_tries) {
  if (!h) return fail(SU3_EINVAL, "su3_set_heatbath: NULL handle");
  if (max_tries < 1 || max_tries > kMaxHeatbathTries)
    return fail(SU3_EINVAL, "su3_set_heatbath: max_tries %d not in [1, %d]", max_tries, kMaxHeatbathTries);
  if (max_tries != h->max_tries) {
    SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_set_heatbath");
    drop_graphs(h);
    if (h->batch) su3_batch_invalidate(h->batch);
    if (h->decomp) su3_decomp_invalidate(h->decomp);
    h->max_tries = max_tries;
  }
  return SU3_OK;
}

int su3_bounds_status(unsigned int* status, int clear) {
  if (!status) return fail(SU3_EINVAL, "su3_bounds_status: NULL status");
  *status = 0u;
#ifdef SU3_BOUNDS_CHECK
  cudaError_t (*const tus[5])(unsigned int*, bool) = {su3k_bounds_status_kernels, su3k_bounds_status_f64, su3k_bounds_status_pair,
                                                        su3k_bounds_status_batch, su3k_bounds_status_decomp};
  for (auto f : tus) {
    unsigned int v = 0u;
    SU3_CUDA(f(&v, clear != 0), "su3_bounds_status");
    *status |= v;
  }
  return SU3_OK;
#else
  (void)clear;
  return fail(SU3_EINVAL, "su3_bounds_status: this library was built without bounds checks");
#endif
}

int su3_set_lanes(su3_handle h, int lanes) {
  if (!h) return fail(SU3_EINVAL, "su3_set_lanes: NULL handle");
  if (is_batch(h) || su3_decomp_active(h))
    return fail(SU3_EINVAL, "su3_set_lanes: not for batch or decomposed handles");
  if (lanes != 0 && lanes != 1 && lanes != 4) return fail(SU3_EINVAL, "su3_set_lanes: lanes %d not 0, 1 or 4", lanes);
  const bool split = lanes == 0 ? use_split(h->geom.Vh, h->precision) : lanes == 4;
  if (split != h->split || lanes != h->lanes) {
    SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_set_lanes");
    drop_graphs(h);
    h->split = split;
    h->lanes = lanes;
  }
  return SU3_OK;
}

int su3_set_schedule(su3_handle h, int schedule) {
  if (!h) return fail(SU3_EINVAL, "su3_set_schedule: NULL handle");
  if (is_batch(h) || su3_decomp_active(h))
    return fail(SU3_EINVAL, "su3_set_schedule: not for batch or decomposed handles");
  if (schedule != SU3_SCHED_AUTO && schedule != SU3_SCHED_PHASES && schedule != SU3_SCHED_PERSISTENT &&
      schedule != SU3_SCHED_PER_DIRECTION && schedule != SU3_SCHED_CHAINED)
    return fail(SU3_EINVAL, "su3_set_schedule: unknown schedule %d", schedule);
  if (!schedule_applies(h, schedule))
    return fail(SU3_EINVAL,
                "su3_set_schedule: the persistent and chained sweeps need one thread per link (pair) and x3 layers "
                "of whole blocks: the site-paired FP32 store (L3 >= 8, the natural block order; all forms) or the "
                "FP64 store (L3 >= 4; per direction or chained half-sweeps)");
  if (schedule != h->schedule) {
    SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_set_schedule");
    drop_graphs(h);
    h->schedule = schedule;
  }
  return SU3_OK;
}

int su3_get_schedule(su3_handle h, int* schedule) {
  if (!h || !schedule) return fail(SU3_EINVAL, "su3_get_schedule: NULL argument");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_get_schedule: batch handle");
  *schedule = su3_decomp_active(h) ? SU3_SCHED_PHASES : effective_schedule(h);
  return SU3_OK;
}

int su3_sweep_debug(su3_handle h, double wait_limit_s, int withhold_item) {
  if (!h) return fail(SU3_EINVAL, "su3_sweep_debug: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_sweep_debug: batch handle (use su3_batch_debug)");
  if (!(wait_limit_s > 0.0) || wait_limit_s > 60.0) return fail(SU3_EINVAL, "su3_sweep_debug: wait limit not in (0, 60] s");
  if (withhold_item < -1) return fail(SU3_EINVAL, "su3_sweep_debug: withhold_item < -1");
  SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_sweep_debug");
  drop_graphs(h);
  h->pq_wait_ns = (long long)(wait_limit_s * 1e9);
  h->pq_withhold = withhold_item;
  return SU3_OK;
}

int su3_set_block_size(su3_handle h, int threads) {
  if (!h) return fail(SU3_EINVAL, "su3_set_block_size: NULL handle");
  if (is_batch(h)) return fail(SU3_EINVAL, "su3_set_block_size: batch handle (use the su3_batch_* calls)");
  const bool set = threads != 0;
  if (!set) threads = default_threads(h->pairs ? h->pgeom.Vh : h->geom.Vh);
  if (threads < 32 || threads > kMaxSweepThreads || (threads & 31))
    return fail(SU3_EINVAL, "su3_set_block_size: %d is not a multiple of 32 in [32, %d]", threads, kMaxSweepThreads);
  if (threads != h->threads || set != h->threads_set) {
    SU3_CUDA(cudaStreamSynchronize(h->stream), "su3_set_block_size");
    drop_graphs(h);
    if (h->decomp) su3_decomp_invalidate(h->decomp);
    h->threads = threads;
    h->threads_set = set;
  }
  return SU3_OK;
}

}  // extern "C"
