// kf_chain_mark.cu -- the kernels of KF_ADAPTIVE's first pass over a chain, one
// per layout.
#include "kf_chain_kernel.cuh"

namespace kf {
int launch_chain_mark(const ChainArgs &a, unsigned blocks, int threads, cudaStream_t s) {
  return launch_chain_by_width<kAdaptive>(a, blocks, threads, s);
}
}  // namespace kf
