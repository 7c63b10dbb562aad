// kf_chain_joseph.cu -- the Joseph-form chain's kernels, one per layout.
#include "kf_chain_kernel.cuh"

namespace kf {
int launch_chain_joseph(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s) {
  return launch_chain_by_width<kJoseph>(a, blocks, threads, s);
}
}  // namespace kf
