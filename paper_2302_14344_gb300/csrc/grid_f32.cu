// The grid kernel's variants with FP32 iterations (the mixed form).
#include "grid_kernel.cuh"
#include "grid_iter.cuh"

namespace subadmm {

KernFn grid_kernel_f32(int split)
{
    return split == 32 ? grid_step_kernel<float, 32> : split == 16 ? grid_step_kernel<float, 16> : grid_step_kernel<float, 8>;
}

KernFn grid_setup_f32() { return grid_setup_kernel<float>; }
KernFn grid_iter_f32(bool wide_rows)
{
    return wide_rows ? grid_iter_kernel<float, true> : grid_iter_kernel<float, false>;
}

}  // namespace subadmm
