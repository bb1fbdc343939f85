// Column CTA solver instantiations (FP64 and mixed), rosenbrock family, n <= 128.
#include "nls_cols_kernels.cuh"

namespace nls {

KernelInfo cols_kernel_rosenbrock(int n, bool mixed)
{
    return mixed ? cols_info<FAM_ROSENBROCK, true>(n) : cols_info<FAM_ROSENBROCK, false>(n);
}

} // namespace nls
