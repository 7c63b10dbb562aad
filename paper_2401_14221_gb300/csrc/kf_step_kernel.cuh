// kf_step_kernel.cuh -- the single step's kernels: one thread per track, and
// its grid-stride form for arrays in host memory.  Instantiated in kf_step.cu
// (float variants) and kf_step_f64.cu (double-arithmetic variants).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kf_device.cuh"
#include "kf_step.cuh"

namespace kf {

struct Loc {
  int64_t base;
  int64_t stride;
};

// Element (c, i) of a C-component array sits at base + c * stride.
template <int C>
__device__ __forceinline__ Loc locate(int64_t i, int64_t n, int32_t soa, int32_t lw) {
  if (soa) return {i, n};
  const int64_t W = int64_t(1) << lw;
  return {(i >> lw) * (C * W) + (i & (W - 1)), W};
}

// Track i of a step launch (i < a.n): load, step, store.
template <int KIND, int VARIANT>
__device__ __forceinline__ void step_track(const StepArgs &a, int64_t i) {
  const Loc l6 = locate<6>(i, a.n, a.soa, a.lw);
  const Loc l21 = locate<21>(i, a.n, a.soa, a.lw);
  const Loc l3 = locate<3>(i, a.n, a.soa, a.lw);

  float p[6], C[21];
#pragma unroll
  for (int c = 0; c < 6; ++c) p[c] = __ldg(a.state_in + l6.base + c * l6.stride);
#pragma unroll
  for (int e = 0; e < 21; ++e) C[e] = __ldg(a.cov_in + l21.base + e * l21.stride);
  const float qf = (float)__ldg(a.charge + i);
  const float surf = __ldg(a.surf + (a.surf_per_track ? i : 0));

  unsigned st;
  if (KIND == kP2z) {
    const float hx = __ldg(a.hit + l3.base);
    const float hy = __ldg(a.hit + l3.base + l3.stride);
    const float vxx = __ldg(a.hitcov + l6.base);
    const float vxy = __ldg(a.hitcov + l6.base + l6.stride);
    const float vyy = __ldg(a.hitcov + l6.base + 2 * l6.stride);
    st = p2z_step<VARIANT>(p, C, qf, a.bz, surf, hx, hy, vxx, vxy, vyy);
  } else {
    const float hx = __ldg(a.hit + l3.base);
    const float hy = __ldg(a.hit + l3.base + l3.stride);
    const float hz = __ldg(a.hit + l3.base + 2 * l3.stride);
    float hc[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) hc[c] = __ldg(a.hitcov + l6.base + c * l6.stride);
    st = p2r_step<VARIANT>(p, C, qf, a.bz, surf, hx, hy, hz, hc);
  }
  if constexpr (VARIANT == kAdaptive) {
    if (st & kRedo) {  // ill-conditioned in FP32: left to the FP64 redo pass
      a.status[i] = (uint8_t)kRedo;
      return;
    }
  }
  st |= finite_status(p, C);

#pragma unroll
  for (int c = 0; c < 6; ++c) __stcs(a.state_out + l6.base + c * l6.stride, p[c]);
#pragma unroll
  for (int e = 0; e < 21; ++e) __stcs(a.cov_out + l21.base + e * l21.stride, C[e]);
  if (a.status) a.status[i] = (uint8_t)st;
}

// Ask L2 for the AoSoA blocks of a C-component array that hold tracks
// [i0, i1): one bulk prefetch of the whole blocks (contiguous, 16-byte
// aligned: the array is, and a block is C * W * 4 bytes with W >= 16).
template <int C>
__device__ __forceinline__ void prefetch_blocks(const float *arr, int64_t i0, int64_t i1,
                                                int32_t lw) {
  const int64_t b0 = i0 >> lw, b1 = (i1 - 1) >> lw;
  const int64_t W = int64_t(1) << lw;
  const uint32_t bytes = (uint32_t)((b1 - b0 + 1) * C * W * 4);
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(arr + b0 * C * W), "r"(bytes)
               : "memory");
}

// One track per thread.  Launched as a programmatic dependent of the
// previous kernel on the stream: it lets the next one be scheduled at once
// and waits for the previous one to complete before it touches memory.
// Under AoSoA a CTA that lands on an SM while the previous kernel drains
// first asks L2 for its inputs -- one bulk prefetch per array of the CTA's
// whole blocks: the state and covariance, for p2r also the hit and hit
// covariance; p2z reads only the first rows of those (x, y and the 2x2
// covariance), so for p2z one prefetch per block of each covers just those
// rows -- so that its loads after the wait find them there instead of in
// HBM.  A prefetch only moves lines
// into L2, where every SM's loads and stores meet, so it cannot return a
// value the previous kernel has yet to write.  Measured on GB300, 960,000
// p2r tracks in graphs of 16 launches: AoSoA 36.6-37.2 -> 35.5 us per
// launch.  Under SoA the same would take one prefetch per component row of
// 512 bytes; that measured slower (37.9 -> 40.0 us) and is not done.
template <int KIND, int VARIANT>
__global__ void __launch_bounds__(256) step_kernel(const __grid_constant__ StepArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x;
  if (!a.soa) {
    const int64_t i1 = i0 + blockDim.x < a.n ? i0 + blockDim.x : a.n;
    if (threadIdx.x == 0) {
      prefetch_blocks<6>(a.state_in, i0, i1, a.lw);
      prefetch_blocks<21>(a.cov_in, i0, i1, a.lw);
      if (KIND == kP2r) {
        prefetch_blocks<3>(a.hit, i0, i1, a.lw);
        prefetch_blocks<6>(a.hitcov, i0, i1, a.lw);
      }
    }
    if (KIND == kP2z) {
      // p2z reads the hit's x, y rows and the covariance's xx, xy, yy rows:
      // the first 2 and 3 rows of each block, one prefetch each per block
      const int64_t W = int64_t(1) << a.lw, b0 = i0 >> a.lw, nb = ((i1 - 1) >> a.lw) - b0 + 1;
      if ((int64_t)threadIdx.x < nb) {
        const int64_t blk = b0 + threadIdx.x;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.hit + blk * 3 * W),
                     "r"((uint32_t)(2 * W * 4))
                     : "memory");
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.hitcov + blk * 6 * W),
                     "r"((uint32_t)(3 * W * 4))
                     : "memory");
      }
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t i = i0 + threadIdx.x;
  if (i < a.n) step_track<KIND, VARIANT>(a, i);
}

// The same as a persistent grid-stride loop, for arrays in host memory: a
// small grid whose warps are at different points of their tracks keeps both
// directions of the CPU-GPU link busy at once, where a grid of n / 256 CTAs
// reads in waves and then writes in waves.  Measured on GB300, 960,000 p2r
// tracks from page-locked memory: one track per thread 0.896 ms; grid-stride
// with 1, 2, 4 CTAs of 256 threads per SM 0.725, 0.758, 0.780 ms; half the
// SMs 0.739 ms; 128-thread CTAs 0.736 ms.
template <int KIND, int VARIANT>
__global__ void __launch_bounds__(256) step_kernel_strided(const __grid_constant__ StepArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride)
    step_track<KIND, VARIANT>(a, i);
}

}  // namespace kf
