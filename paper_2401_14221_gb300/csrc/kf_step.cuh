// kf_step.cuh -- arguments of the single-step kernel and its launcher,
// shared by the device-pointer and host-pointer entry points.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kf_device.cuh"

namespace kf {

// Device pointers and sizes for one single-step launch (already validated).
struct StepArgs {
  const float *state_in;
  const float *cov_in;
  float *state_out;
  float *cov_out;
  const int8_t *charge;
  const float *hit;
  const float *hitcov;
  const float *surf;
  uint8_t *status;  // may be NULL
  int64_t n;
  int32_t soa;  // 1: [C][n] arrays; 0: AoSoA blocks of 2^lw tracks
  int32_t lw;
  float bz;
  int32_t surf_per_track;
  unsigned *err = nullptr;  // device error word (set by the staged launcher)
  // Polls of a staged-pipeline barrier by a compute warp before it gives up
  // (set by the staged launcher from kf_set_device_wait_limit).
  uint32_t wait_polls = 0;
};

#ifdef __CUDACC__
// Status bytes base .. base+15 of an [n] array as four little-endian words:
// one 16-byte load where the array is 16-byte aligned and the run is whole,
// byte loads otherwise (bytes at or past n read as 0).
__device__ __forceinline__ uint4 load_status16(const uint8_t *status, int64_t base, int64_t n) {
  if (base + 16 <= n && (reinterpret_cast<uintptr_t>(status) & 15u) == 0)
    return *reinterpret_cast<const uint4 *>(status + base);
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if (base + j < n) w[j >> 2] |= (uint32_t)status[base + j] << (8 * (j & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Redo passes gather the marked tracks of a span of kRedoSpan tracks into a
// shared-memory list before running them, so that each warp runs up to 32
// marked tracks instead of one marked track among 31 idle lanes: GB300
// issues an FP64 warp instruction over 64 cycles whether or not its lanes
// are active.  A block has one warp per scheduler, and a span is small enough
// that its marks rarely take it a second round and large enough that the
// blocks leave the next step's room to start prefetching while this pass
// looks through the marks (us per p2r step, spans / threads 4,096/128,
// 2,048/128, 2,048/64, 4,096/64: 960,000 tracks with nothing marked 37.1,
// 37.9, 37.1, 37.7; with 3 % marked 54.9, 65.4, 60.4, 61.3; 300,007: 30.2,
// 29.5, 30.0, 35.0).
constexpr int kRedoSpan = 4096;
constexpr int kRedoThreads = 128;

// A redo pass is a programmatic dependent of its step: it waits here until that
// has completed and its status marks are visible.  It lets the next kernel on
// the stream be scheduled before the wait where the step fills the device (that
// kernel then sets up and asks L2 for its inputs while this pass runs, and waits
// for it before it reads or writes anything), after it where step, pass and the
// next step are on the device together anyway: there the next step's blocks, let
// in early, keep the pass after them waiting for room.  us per step with nothing
// marked, three batches in turn, before and after the wait: p2z 20,000 tracks
// 4.22 and 3.40, 60,000 5.76 and 4.49, 100,000 6.68 and 5.45, 130,000 6.95 and
// 6.27, 200,000 9.31 and 10.36; p2r 60,000 6.19 and 5.11, 130,000 7.50 and 7.43,
// 200,000 10.4 and 11.8, 960,000 37.4 and 38.4.
constexpr int64_t kRedoEarlyTracks = 1 << 17;
__device__ __forceinline__ void redo_wait(int64_t n) {
  const bool early = n > kRedoEarlyTracks;
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Fill list[0..count) with the offsets (from span0) of the tracks marked
// kRedo among [span0, min(span0 + SPAN, n)); returns the count.  Every
// thread of the block (THREADS of them) must call it.  Each thread looks at
// SPAN / (16 THREADS) runs of 16 status bytes, all loaded before any is
// examined, so a span with nothing marked costs one memory latency.
template <int SPAN, int THREADS>
__device__ __forceinline__ int gather_marked(const uint8_t *status, int64_t span0, int64_t n,
                                             uint16_t *list, int *count) {
  constexpr int kRuns = SPAN / (16 * THREADS);
  static_assert(kRuns * 16 * THREADS == SPAN, "whole runs per thread");
  static_assert(SPAN <= 65536, "span offsets are 16-bit");
  constexpr uint32_t kMarks = 0x01010101u * kRedo;  // the kRedo bit of each byte
  if (threadIdx.x == 0) *count = 0;
  uint4 v[kRuns];
#pragma unroll
  for (int r = 0; r < kRuns; ++r) {
    const int64_t base = span0 + (int64_t)(r * THREADS + threadIdx.x) * 16;
    v[r] = base < n ? load_status16(status, base, n) : make_uint4(0u, 0u, 0u, 0u);
  }
  __syncthreads();  // count is 0
#pragma unroll
  for (int r = 0; r < kRuns; ++r) {
    const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    if (((w[0] | w[1] | w[2] | w[3]) & kMarks) == 0u) continue;
    const int off = (r * THREADS + (int)threadIdx.x) * 16;
    for (int j = 0; j < 16; ++j)
      if ((w[j >> 2] >> (8 * (j & 3))) & kRedo) list[atomicAdd(count, 1)] = (uint16_t)(off + j);
  }
  __syncthreads();
  return *count;
}

#endif

// How a step (or chain) launch is shaped.
struct LaunchConfig {
  int kernel;       // KF_STEP_DIRECT or KF_STEP_STAGED
  int threads;      // CTA size of the one-thread-per-track kernels
  int ctas_per_sm;  // persistent CTAs per SM of the staged kernel
};

// Launch the p2z (kind 0) or p2r (kind 1) step kernel for `a` on stream s
// with the given KF_* precision variant.  The shape comes from, in order:
// the autotuner's per-thread override while it measures, the process-wide
// kf_set_step_kernel mode, the tuning cache, the defaults.  plain_loads
// (arrays in host or managed memory) overrides all of them: the
// one-thread-per-track kernel, 256 threads per CTA.
int launch_step_kernel(int kind, int precision, const StepArgs &a, cudaStream_t s,
                       bool plain_loads = false);

// Launches of the one-thread-per-track kernels with the double-arithmetic
// variants (KF_FP64, KF_FP64_UPDATE): on device arrays with the shape lc, and
// on host arrays with a grid of that many 256-thread CTAs.
cudaError_t launch_direct_f64(int kind, int precision, const StepArgs &a,
                              const cudaLaunchConfig_t &lc);
void launch_strided_f64(int kind, int precision, const StepArgs &a, unsigned grid,
                        cudaStream_t s);

// Second pass of KF_ADAPTIVE: redo in FP64 every track whose status the
// step kernel marked with kRedo (those tracks' outputs are not yet written).
int launch_redo_pass(int kind, const StepArgs &a, cudaStream_t s);

// The persistent bulk-async-staged kernel (AoSoA layouts only).
int launch_step_staged(int kind, int precision, const StepArgs &a, cudaStream_t s,
                       int ctas_per_sm);

// Process-wide choice between the kernels: KF_STEP_AUTO / _DIRECT / _STAGED.
int step_kernel_mode();

// Whether a chain of n tracks runs with four warps to 32 tracks on a device of
// that many SMs: one launch shape, kSharedChainThreads a CTA, nothing to tune.
constexpr int kSharedChainThreads = 128;
bool chain_shares_warps(int precision, int64_t n, int sms);

// ------------------------------------------------------------- tuning
enum TuneOp : int { kOpStep = 0, kOpChain = 1 };

// Shape forced on the calling thread's launches (the autotuner sets it
// while it measures candidates); nullptr when none.
const LaunchConfig *thread_override();
void set_thread_override(const LaunchConfig *cfg);

// Cached best shape for (current device, op, kind, precision, layout, n).
bool tune_lookup(int op, int kind, int precision, int soa, int lw, int64_t n, LaunchConfig *out);
void tune_store(int op, int kind, int precision, int soa, int lw, int64_t n,
                const LaunchConfig &cfg, float ms);

}  // namespace kf
