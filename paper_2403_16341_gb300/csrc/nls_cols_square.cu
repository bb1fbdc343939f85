// Column CTA solver instantiations (FP64 and mixed), square family, n <= 128.
#include "nls_cols_kernels.cuh"

namespace nls {

KernelInfo cols_kernel_square(int n, bool mixed)
{
    return mixed ? cols_info<FAM_SQUARE, true>(n) : cols_info<FAM_SQUARE, false>(n);
}

} // namespace nls
