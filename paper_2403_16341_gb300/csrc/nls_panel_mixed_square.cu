// Column-panel CTA solver instantiations: mixed, square family, n <= 32, 64, 96.
#include "nls_panel_kernels.cuh"

namespace nls {

KernelInfo panel_kernel_mixed_square(int n) { return panel_info_for<FAM_SQUARE, true>(n); }

} // namespace nls
