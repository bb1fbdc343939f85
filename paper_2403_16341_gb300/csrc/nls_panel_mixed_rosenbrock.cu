// Column-panel CTA solver instantiations: mixed, rosenbrock family, n <= 32, 64, 96.
#include "nls_panel_kernels.cuh"

namespace nls {

KernelInfo panel_kernel_mixed_rosenbrock(int n) { return panel_info_for<FAM_ROSENBROCK, true>(n); }

} // namespace nls
