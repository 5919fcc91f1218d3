// FP32 instantiations of the grouped regime (i) kernel for an A that a tensor
// map cannot describe, in each load form.
#include "tsmm_group.cuh"

namespace tsmm {
cudaError_t launch_grouped_async_f32(int np, int lv, const GroupParams &gp, cudaStream_t s) {
    return launch_grouped_async_dispatch<float>(np, lv, gp, s);
}
}  // namespace tsmm
