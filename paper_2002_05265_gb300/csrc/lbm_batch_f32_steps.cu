// Batched persistent sweep kernels, one step at a time, for float population storage, one per (VEC, BLOCK) shape
// the autotuner may choose.
#include "lbm_batch.cuh"
#include "lbm_internal.h"

namespace lbm {
const void* batch_kernel_f32_steps(int vec, int block) {
    if (vec == 4 && block == 256) return (const void*)batch_kernel<float, 4, 256, false>;
    if (vec == 4 && block == 128) return (const void*)batch_kernel<float, 4, 128, false>;
    if (vec == 4 && block == 512) return (const void*)batch_kernel<float, 4, 512, false>;
    if (vec == 2 && block == 256) return (const void*)batch_kernel<float, 2, 256, false>;
    if (vec == 2 && block == 128) return (const void*)batch_kernel<float, 2, 128, false>;
    if (vec == 2 && block == 512) return (const void*)batch_kernel<float, 2, 512, false>;
    return nullptr;
}
}  // namespace lbm
