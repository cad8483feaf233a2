// The grid kernel's variants with FP64 iterations.
#include "grid_kernel.cuh"
#include "grid_iter.cuh"

namespace subadmm {

KernFn grid_kernel_f64(int split)
{
    return split == 32 ? grid_step_kernel<double, 32> : split == 16 ? grid_step_kernel<double, 16> : grid_step_kernel<double, 8>;
}

KernFn grid_setup_f64() { return grid_setup_kernel<double>; }
KernFn grid_iter_f64(bool wide_rows)
{
    return wide_rows ? grid_iter_kernel<double, true> : grid_iter_kernel<double, false>;
}

}  // namespace subadmm
