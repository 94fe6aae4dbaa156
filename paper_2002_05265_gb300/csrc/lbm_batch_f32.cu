// Batched persistent sweep kernels for float population storage, one per (VEC, BLOCK) shape
// the autotuner may choose.
#include "lbm_batch.cuh"
#include "lbm_internal.h"

namespace lbm {
const void* batch_kernel_f32(int vec, int block, bool fused) {
    if (!fused) return batch_kernel_f32_steps(vec, block);
    if (vec == 4 && block == 256) return (const void*)batch_kernel<float, 4, 256, true>;
    if (vec == 4 && block == 128) return (const void*)batch_kernel<float, 4, 128, true>;
    if (vec == 4 && block == 512) return (const void*)batch_kernel<float, 4, 512, true>;
    if (vec == 2 && block == 256) return (const void*)batch_kernel<float, 2, 256, true>;
    if (vec == 2 && block == 128) return (const void*)batch_kernel<float, 2, 128, true>;
    if (vec == 2 && block == 512) return (const void*)batch_kernel<float, 2, 512, true>;
    return nullptr;
}
}  // namespace lbm
