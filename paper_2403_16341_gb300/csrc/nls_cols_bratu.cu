// Column CTA solver instantiations (FP64 and mixed), bratu family, n <= 128.
#include "nls_cols_kernels.cuh"

namespace nls {

KernelInfo cols_kernel_bratu(int n, bool mixed)
{
    return mixed ? cols_info<FAM_BRATU, true>(n) : cols_info<FAM_BRATU, false>(n);
}

} // namespace nls
