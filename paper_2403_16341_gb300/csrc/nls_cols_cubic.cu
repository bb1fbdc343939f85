// Column CTA solver instantiations (FP64 and mixed), cubic family, n <= 128.
#include "nls_cols_kernels.cuh"

namespace nls {

KernelInfo cols_kernel_cubic(int n, bool mixed)
{
    return mixed ? cols_info<FAM_CUBIC, true>(n) : cols_info<FAM_CUBIC, false>(n);
}

} // namespace nls
