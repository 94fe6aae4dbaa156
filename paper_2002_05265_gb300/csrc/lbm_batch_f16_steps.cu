// Batched persistent sweep kernels, one step at a time, for __half population storage, one per (VEC, BLOCK) shape
// the autotuner may choose.
#include "lbm_batch.cuh"
#include "lbm_internal.h"

namespace lbm {
const void* batch_kernel_f16_steps(int vec, int block) {
    if (vec == 8 && block == 512) return (const void*)batch_kernel<__half, 8, 512, false>;
    if (vec == 8 && block == 256) return (const void*)batch_kernel<__half, 8, 256, false>;
    if (vec == 8 && block == 128) return (const void*)batch_kernel<__half, 8, 128, false>;
    if (vec == 4 && block == 256) return (const void*)batch_kernel<__half, 4, 256, false>;
    if (vec == 4 && block == 128) return (const void*)batch_kernel<__half, 4, 128, false>;
    return nullptr;
}
}  // namespace lbm
