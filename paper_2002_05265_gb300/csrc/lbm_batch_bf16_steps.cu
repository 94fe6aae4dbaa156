// Batched persistent sweep kernels, one step at a time, for __nv_bfloat16 population storage, one per (VEC, BLOCK) shape
// the autotuner may choose.
#include "lbm_batch.cuh"
#include "lbm_internal.h"

namespace lbm {
const void* batch_kernel_bf16_steps(int vec, int block) {
    if (vec == 8 && block == 512) return (const void*)batch_kernel<__nv_bfloat16, 8, 512, false>;
    if (vec == 8 && block == 256) return (const void*)batch_kernel<__nv_bfloat16, 8, 256, false>;
    if (vec == 8 && block == 128) return (const void*)batch_kernel<__nv_bfloat16, 8, 128, false>;
    if (vec == 4 && block == 256) return (const void*)batch_kernel<__nv_bfloat16, 4, 256, false>;
    if (vec == 4 && block == 128) return (const void*)batch_kernel<__nv_bfloat16, 4, 128, false>;
    return nullptr;
}
}  // namespace lbm
