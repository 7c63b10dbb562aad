// kf_chain_df.cu -- the chain's kernels with the double-float update, one per
// layout.
#include "kf_chain_kernel.cuh"

namespace kf {
int launch_chain_df(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s) {
  return launch_chain_by_width<kDFUpdate>(a, blocks, threads, s);
}
}  // namespace kf
