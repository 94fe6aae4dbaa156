// Time-fused step kernels for __half population storage.
#include "lbm_march.cuh"
#include "lbm_internal.h"

namespace lbm {
template <bool SHIFT, bool PAIRS>
static const void* march_table(bool roll) {
    return roll ? (const void*)march_kernel<__half, SHIFT, PAIRS, true> : (const void*)march_kernel<__half, SHIFT, PAIRS, false>;
}
const void* march_kernel_f16(bool shifted, bool pairs, bool roll) {
    if (pairs) return shifted ? march_table<true, true>(roll) : march_table<false, true>(roll);
    return shifted ? march_table<true, false>(roll) : march_table<false, false>(roll);
}
}  // namespace lbm
