// kf_chain_kernel.cuh -- the chain kernel and its launch by layout.
#pragma once

#include <cstdint>

#include "kf_common.cuh"
#include "kf_chain.cuh"
#include "kf_device.cuh"

namespace kf {

struct ChainArgs {
  float *state;
  float *cov;
  const int8_t *charge;
  const float *hits;     // [L] arrays of 3 components in the layout
  const float *hitcovs;  // [L] arrays of 6 components in the layout
  uint8_t *status;
  int64_t n;
  int64_t hit_stride;  // floats between consecutive layers' hit arrays
  int64_t hc_stride;   // floats between consecutive layers' hit-cov arrays
  int32_t soa;
  int32_t lw;
  float bz;
  int32_t L;
  int32_t kinds[KF_MAX_LAYERS];
  float pos[KF_MAX_LAYERS];
  // where KF_ADAPTIVE's first pass lists the tracks it marks (NULL: status
  // marks only)
  uint32_t *redo_count = nullptr;
  uint32_t *redo_list = nullptr;
};

// Track i of the chain: load, run every layer, store.
// LW: the AoSoA block width's logarithm, -1 for SoA, or 0 where a.soa and a.lw
// say.
template <int VARIANT, int LW>
__device__ __forceinline__ void chain_one(const ChainArgs &a, int64_t i) {
  const int32_t soa = LW > 0 ? 0 : LW < 0 ? 1 : a.soa, lw = LW > 0 ? LW : a.lw;
  const ChainLoc l6 = chain_locate<6>(i, a.n, soa, lw);
  const ChainLoc l21 = chain_locate<21>(i, a.n, soa, lw);
  const ChainLoc l3 = chain_locate<3>(i, a.n, soa, lw);

  float p[6], C[21];
#pragma unroll
  for (int c = 0; c < 6; ++c) p[c] = a.state[l6.base + c * l6.stride];
#pragma unroll
  for (int e = 0; e < 21; ++e) C[e] = a.cov[l21.base + e * l21.stride];
  const float qf = (float)__ldg(a.charge + i);

  unsigned st;
  if constexpr (VARIANT == kAdaptive) {
    st = chain_track_marking(p, C, qf, a.bz, a.L, a.kinds, a.pos, a.hits, a.hit_stride, a.hitcovs,
                             a.hc_stride, l3, l6);
    if (st & kRedo) {  // left to the second pass, inputs untouched
      a.status[i] = (uint8_t)kRedo;
      if (a.redo_list) a.redo_list[atomicAdd(a.redo_count, 1u)] = (uint32_t)i;
      return;
    }
  } else if constexpr (VARIANT == kFP64) {
    st = chain_track_fp64(p, C, qf, a.bz, a.L, a.kinds, a.pos, a.hits, a.hit_stride, a.hitcovs,
                          a.hc_stride, l3, l6);
  } else {
    st = chain_track<VARIANT>(p, C, qf, a.bz, a.L, a.kinds, a.pos, a.hits, a.hit_stride,
                              a.hitcovs, a.hc_stride, l3, l6);
  }
  st |= finite_status(p, C);
#pragma unroll
  for (int c = 0; c < 6; ++c) a.state[l6.base + c * l6.stride] = p[c];
#pragma unroll
  for (int e = 0; e < 21; ++e) a.cov[l21.base + e * l21.stride] = C[e];
  if (a.status) a.status[i] = (uint8_t)st;
}

// One track per thread.  KF_ADAPTIVE's first pass is the same kernel (kAdaptive:
// marked tracks are left alone).  The float variants take 80 registers: 72 and
// 64 spill and lose 1 to 6 %, 88 gain nothing.
template <int VARIANT, int LW>
__global__ void __launch_bounds__(256)
    chain_kernel(const __grid_constant__ ChainArgs a) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.n) chain_one<VARIANT, LW>(a, i);
}

// The kernel with the AoSoA width known at compile time: a hit's nine loads
// then differ by immediate offsets, which takes 4 % of the chain's instructions
// and the 64-bit strides out of its registers (1.75 M tracks, FP32 391 -> 381
// us, Joseph 467 -> 455, double-float update 838 -> 817, adaptive 605 -> 582).
// SoA gets a kernel too, but for the double-float update, whose SoA kernel
// spills (860 us; 838 with strides known at run time).
template <int VARIANT>
int launch_chain_by_width(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s) {
  constexpr int kSoa = VARIANT == kDFUpdate ? 0 : -1;
  switch (a.soa ? -1 : a.lw) {
    case 4: chain_kernel<VARIANT, 4><<<blocks, threads, 0, s>>>(a); break;
    case 5: chain_kernel<VARIANT, 5><<<blocks, threads, 0, s>>>(a); break;
    case 6: chain_kernel<VARIANT, 6><<<blocks, threads, 0, s>>>(a); break;
    case 7: chain_kernel<VARIANT, 7><<<blocks, threads, 0, s>>>(a); break;
    default: chain_kernel<VARIANT, kSoa><<<blocks, threads, 0, s>>>(a); break;
  }
  return check_cuda(cudaGetLastError(), "chain launch");
}

// Instantiated in units of their own (kf_chain_fp32.cu, kf_chain_joseph.cu,
// kf_chain_df.cu, kf_chain_mark.cu).
int launch_chain_fp32(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s);
int launch_chain_joseph(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s);
int launch_chain_df(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s);
int launch_chain_mark(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s);

}  // namespace kf
