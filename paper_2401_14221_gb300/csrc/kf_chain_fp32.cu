// kf_chain_fp32.cu -- the FP32 chain's kernels, one per layout.
#include "kf_chain_kernel.cuh"

namespace kf {
int launch_chain_fp32(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s) {
  return launch_chain_by_width<kFP32>(a, blocks, threads, s);
}
}  // namespace kf
