// kf_step_f64.cu -- the single step's kernels with the double-arithmetic
// variants (FP64 update, all-FP64), built like the staged kernel's of the same
// variants so that all of them round alike, denormals included.
#include "kf_common.cuh"
#include "kf_step_kernel.cuh"

namespace kf {

cudaError_t launch_direct_f64(int kind, int precision, const StepArgs &a,
                              const cudaLaunchConfig_t &lc) {
  if (kind == kP2z)
    return precision == KF_FP64 ? cudaLaunchKernelEx(&lc, step_kernel<kP2z, kFP64>, a)
                                : cudaLaunchKernelEx(&lc, step_kernel<kP2z, kFP64Update>, a);
  return precision == KF_FP64 ? cudaLaunchKernelEx(&lc, step_kernel<kP2r, kFP64>, a)
                              : cudaLaunchKernelEx(&lc, step_kernel<kP2r, kFP64Update>, a);
}

void launch_strided_f64(int kind, int precision, const StepArgs &a, unsigned grid,
                        cudaStream_t s) {
  if (kind == kP2z) {
    if (precision == KF_FP64) step_kernel_strided<kP2z, kFP64><<<grid, 256, 0, s>>>(a);
    else step_kernel_strided<kP2z, kFP64Update><<<grid, 256, 0, s>>>(a);
  } else {
    if (precision == KF_FP64) step_kernel_strided<kP2r, kFP64><<<grid, 256, 0, s>>>(a);
    else step_kernel_strided<kP2r, kFP64Update><<<grid, 256, 0, s>>>(a);
  }
}

}  // namespace kf
