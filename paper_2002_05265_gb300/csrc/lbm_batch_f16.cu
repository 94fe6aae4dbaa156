// Batched persistent sweep kernels for __half population storage, one per (VEC, BLOCK) shape
// the autotuner may choose.
#include "lbm_batch.cuh"
#include "lbm_internal.h"

namespace lbm {
const void* batch_kernel_f16(int vec, int block, bool fused) {
    if (!fused) return batch_kernel_f16_steps(vec, block);
    if (vec == 8 && block == 512) return (const void*)batch_kernel<__half, 8, 512, true>;
    if (vec == 8 && block == 256) return (const void*)batch_kernel<__half, 8, 256, true>;
    if (vec == 8 && block == 128) return (const void*)batch_kernel<__half, 8, 128, true>;
    if (vec == 4 && block == 256) return (const void*)batch_kernel<__half, 4, 256, true>;
    if (vec == 4 && block == 128) return (const void*)batch_kernel<__half, 4, 128, true>;
    return nullptr;
}
}  // namespace lbm
