// Instantiations of the CE kernel for FP64 jobs with 4 trials per
// thread (one translation unit per fold mode and trials per thread, so that
// they compile in parallel).
#include "gce_kernel.cuh"

namespace gce {

const void *main_kernel_ptr_fp64_t4(int block, int kv) {
    return kernel_for_variant<kJobFp64, 4>(block, kv);
}

cudaError_t launch_main_fp64_t4(int block, int grid, size_t smem, const MainArgs &a,
                                  cudaStream_t s) {
    return launch_for_block<kJobFp64, 4>(block, grid, smem, a, s);
}

}  // namespace gce
