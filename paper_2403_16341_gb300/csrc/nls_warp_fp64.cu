// Warp-tiled solver instantiations (fp64), L = 8, 16, 32 lanes per instance.
#include "nls_internal.h"
#include "nls_warp.cuh"

namespace nls {

template <int L, int FAM>
static cudaError_t launch_warp_fp64(const SolveArgs &a, int grid, cudaStream_t st)
{
    k_solve_warp<L, FAM, false><<<grid, (warp_tpb<L, FAM, false>()), warp_smem_bytes<L, false, FAM>(), st>>>(a);
    return cudaGetLastError();
}

template <int L, int FAM>
static KernelInfo info_fp64()
{
    KernelInfo k;
    k.launch = &launch_warp_fp64<L, FAM>;
    k.func = reinterpret_cast<const void *>(&k_solve_warp<L, FAM, false>);
    k.block = warp_tpb<L, FAM, false>();
    k.smem = warp_smem_bytes<L, false, FAM>();
    // An SM's split between L1 and shared memory changes only when the SM is idle,
    // and the driver takes the smallest split that a kernel's occupancy needs.
    // Beside a 32-lane kernel of another family, which needs half of what the cubic
    // does, the cubic's CTAs then waited for it to drain (one flush, Bratu n = 32,
    // 664 systems, then cubic n = 32, 279: 627 us, 321 in the other order).  With
    // one split for all 32-lane kernels: 321 us in both.
    k.widest_smem = L == 32;
    k.per_cta = (warp_tpb<L, FAM, false>() / 32) * (32 / L);
    return k;
}

template <int L>
static KernelInfo by_family_fp64(int family)
{
    switch (family) {
    case FAM_CUBIC: return info_fp64<L, FAM_CUBIC>();
    case FAM_BRATU: return info_fp64<L, FAM_BRATU>();
    case FAM_SQUARE: return info_fp64<L, FAM_SQUARE>();
    case FAM_ROSENBROCK: return info_fp64<L, FAM_ROSENBROCK>();
    default: return KernelInfo{};
    }
}

KernelInfo warp_kernel_fp64(int family, int L)
{
    switch (L) {
    case 8: return by_family_fp64<8>(family);
    case 16: return by_family_fp64<16>(family);
    case 32: return by_family_fp64<32>(family);
    default: return KernelInfo{};
    }
}

} // namespace nls
