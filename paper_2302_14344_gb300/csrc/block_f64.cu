// The block kernel's variants with FP64 iterations.
#include "step_kernel.cuh"

namespace subadmm {

KernFn block_kernel_f64(bool cached, int split, int nt)
{
    if (cached) return split == 4 ? step_kernel<double, 4, true> : split == 2 ? step_kernel<double, 2, true> : step_kernel<double, 1, true>;
    if (nt == SUBADMM_WIDE)
        return split == 4 ? step_kernel<double, 4, false, SUBADMM_WIDE>
             : split == 2 ? step_kernel<double, 2, false, SUBADMM_WIDE>
                          : step_kernel<double, 1, false, SUBADMM_WIDE>;
    return split == 4 ? step_kernel<double, 4, false> : split == 2 ? step_kernel<double, 2, false> : step_kernel<double, 1, false>;
}

}  // namespace subadmm
