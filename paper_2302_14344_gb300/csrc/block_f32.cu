// The block kernel's variants with FP32 iterations (the mixed form).
#include "step_kernel.cuh"

namespace subadmm {

KernFn block_kernel_f32(bool cached, int split, int nt)
{
    if (cached) return split == 4 ? step_kernel<float, 4, true> : split == 2 ? step_kernel<float, 2, true> : step_kernel<float, 1, true>;
    if (nt == SUBADMM_WIDE)
        return split == 4 ? step_kernel<float, 4, false, SUBADMM_WIDE>
             : split == 2 ? step_kernel<float, 2, false, SUBADMM_WIDE>
                          : step_kernel<float, 1, false, SUBADMM_WIDE>;
    return split == 4 ? step_kernel<float, 4, false> : split == 2 ? step_kernel<float, 2, false> : step_kernel<float, 1, false>;
}

}  // namespace subadmm
