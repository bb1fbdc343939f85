// nls_internal.h -- host-side registry of the solver kernels.
#pragma once

#include <cuda_runtime.h>

#include "nls_common.cuh"

namespace nls {

using LaunchFn = cudaError_t (*)(const SolveArgs &, int grid, cudaStream_t);

struct KernelInfo {
    LaunchFn launch = nullptr;
    const void *func = nullptr;
    int block = 0;     // threads per CTA
    int smem = 0;      // dynamic shared memory bytes
    int smem_most = 0; // most dynamic shared memory of any launch of func, where that is above 48 KB for some n
    bool widest_smem = false; // an SM running it is configured for the most shared memory
    int per_cta = 0;   // instances per CTA per round (static grids)
};

// Refill threshold of a persistent thread-tiled grid when the caller set none
// (a warp refills its idle lanes when at most this many still iterate).  A
// refill of a few lanes costs a whole warp's initial residual, idle lanes cost
// their share of every pass: few lanes left is the better point where pass
// counts are close together (2^19 cubic n = 8, from 24 to 8: Newton FP64 2.58 ->
// 2.44 ms, mixed 1.21 -> 0.98; backtracking 2.94 -> 2.62 and 1.56 -> 1.19; trust
// region 3.43 -> 3.37 and 1.30 -> 1.27; Bratu n = 8 4 to 15%; square within 1%),
// early refills where they spread widely (Rosenbrock n = 8, trust region: 11.6
// ms with 24, 14.2 with 8).
// Potra-Ptak, a local method that can wander, keeps 24 too (mixed cubic n = 8:
// 2.01 ms, 2.09 with 8).
inline int refill_rule(int family, int alg) { return family == FAM_ROSENBROCK || alg == ALG_POTRA_PTAK ? 24 : 8; }

// One instance per thread, compile-time n in 1..8.
KernelInfo thread_kernel(int family, int n, bool mixed, bool analytic);

// Record a handle-free error message for nls_last_error(NULL); returns code.
int set_global_error(int code, const char *msg);

} // namespace nls

namespace nls {
// One instance per warp segment of L = 8, 16 or 32 lanes (the smallest L >= n,
// or `lanes` when non-zero), runtime n <= L.
KernelInfo warp_kernel(int family, int n, bool mixed, int lanes = 0);
} // namespace nls

namespace nls {
// One instance per CTA, n <= 128: the matrix by columns in shared memory
// (nls_cols.cuh); block and shared memory depend on n.
KernelInfo cta_kernel(int family, int n, bool mixed);
// ... or, in mixed precision and n <= 96, in registers (nls_panel.cuh).
KernelInfo panel_kernel(int family, int n);

// The most mixed-precision instances, over all CTA-tiled requests of a flush, that
// run on panel_kernel.  It has the lower latency, cta_kernel the throughput, so the
// line is one wave of its CTAs (4 per SM up to n = 64, 2 up to n = 96; above that
// the two are within 5%).  Trust region, time here / time of cta_kernel at a wave's
// end and beyond: Bratu n = 64 608: 0.80, 1,000: 1.20; n = 48 0.89, 1.30; n = 96 304:
// 0.91, 456: 1.37; cubic n = 96 0.76, 1.23.  The cubic up to n = 64 re-reads A with
// more threads per instance here, and stays ahead for more waves: n = 33 1,000: 0.91,
// 2,000: 1.07; n = 48 2,000: 0.95, 4,000: 1.03; n = 64 2,000: 0.93, 3,000: 0.94,
// 4,000: 0.99;
// refined n = 48 and 64 1,000: 0.90 and 0.86, 2,000: 1.05 and 1.00; n = 32 2,000: 0.93,
// n = 24 608: 0.69, 1,000: 1.12.  The smallest systems (refined, or asked for) are one
// panel there and gain nothing: 50 systems of n = 8 0.91 (cubic) and 1.03 (Bratu),
// n = 16 0.73 and 0.86.
// In a flush of several requests the cubic's larger sizes stay on the panels for
// four waves (1,024 of n = 40..70 1.02 ms, 1.11 with n > 64 on the columns).
constexpr int PANEL_NMAX = 96;
inline int64_t panel_most(int family, int n, bool refine, bool several, int sms)
{
    const bool cubic = family == FAM_CUBIC;
    if (n > PANEL_NMAX || n < (cubic ? 8 : 9)) return 0;
    const int waves = !cubic || n < 32 ? 1 : n > 64 ? (several ? 4 : 1) : refine || n <= 40 ? 2 : 5;
    return (int64_t)waves * (n <= 64 ? 4 : 2) * sms;
}
} // namespace nls

namespace nls {
// Adjoint sensitivity kernels: one instance per thread (n <= 8), ...
cudaError_t launch_adjoint(int family, int n, const double *params, const double *u, const double *w,
                           double *grad, int32_t *status, int64_t batch, cudaStream_t st);
// ... per warp segment (n <= 32) or per CTA (n <= 128).
cudaError_t launch_adjoint_tiles(int family, int n, const double *params, const double *u, const double *w,
                                 double *grad, int32_t *status, int64_t batch, cudaStream_t st);
} // namespace nls

namespace nls {
// Poly-algorithm helpers (nls_poly.cu).
struct PolyGatherArgs {
    int64_t batch;               // full batch (also the compact arrays' leading dimension)
    int E, n;
    const int32_t *status;       // [batch] statuses after the previous stage
    const double *params;        // [E][batch]
    const double *u0;            // [n][batch] original starting points
    int64_t *idx;                // [batch] compact position -> instance
    double *cparams, *cu;        // [E][batch], [n][batch] compact copies
    unsigned long long *count;   // number gathered (zeroed before)
};
struct PolyScatterArgs {
    int64_t batch;
    int n;
    const unsigned long long *count;
    const int64_t *idx;
    const double *cu;
    const int32_t *cstatus, *citers, *cnfev;
    const double *cresid;
    double *u;
    int32_t *status, *iters, *nfev;
    double *resid;
};
cudaError_t launch_poly_gather(const PolyGatherArgs &g, cudaStream_t st);
cudaError_t launch_poly_scatter(const PolyScatterArgs &s, cudaStream_t st);
cudaError_t launch_poly_total(unsigned long long *solved, const unsigned long long *ctr, int stages,
                              cudaStream_t st);
// Potra-Ptak, Halley, Broyden and modified Broyden (alg = ALG_POTRA_PTAK ..
// ALG_MOD_BROYDEN): one instance per thread (n <= 8), per warp segment of
// L = 16 or 32 lanes, or per CTA (n <= 128).
KernelInfo thread_ext_kernel(int family, int n, int alg, bool mixed);
KernelInfo warp_ext_kernel(int family, int L, int alg, bool mixed);
KernelInfo cta_ext_kernel(int family, int n, int alg, bool mixed);
} // namespace nls
