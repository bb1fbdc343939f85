// nls_cols_kernels.cuh -- launch helpers and registry entries of the
// shared-memory column solver (nls_cols.cuh): one instance per CTA, n <= 128;
// the block and the shared memory follow n.
#pragma once

#include "nls_cols.cuh"
#include "nls_internal.h"

namespace nls {

template <int FAM, bool MIXED>
static cudaError_t launch_cols(const SolveArgs &a, int grid, cudaStream_t st)
{
    constexpr int C = col_panel<MIXED>();
    k_solve_cols<C, FAM, MIXED><<<grid, 32 * col_warps<MIXED>(a.n), col_smem_bytes<C, MIXED>(a.n), st>>>(a);
    return cudaGetLastError();
}

template <int FAM, bool MIXED>
static KernelInfo cols_info(int n)
{
    if (n < 1 || n > COL_NMAX) return KernelInfo{};
    constexpr int C = col_panel<MIXED>();
    KernelInfo k;
    k.launch = &launch_cols<FAM, MIXED>;
    k.func = reinterpret_cast<const void *>(&k_solve_cols<C, FAM, MIXED>);
    k.block = 32 * col_warps<MIXED>(n);
    k.smem = col_smem_bytes<C, MIXED>(n);
    k.smem_most = col_smem_bytes<C, MIXED>(COL_NMAX);
    // One split of an SM's memory for every n: each size needs another amount of
    // shared memory, and an SM changes its split only when it is idle, so in a flush
    // of several sizes the kernels waited for one another (1,024 Bratu systems by
    // trust region, n = 33..50 567 -> 443 us, n = 64..128 1,824 -> 1,575 mixed, 6.05 ->
    // 5.80 ms FP64; 4,096 of n = 40..80 1,744 -> 1,610 us).  Not the cubic, which
    // re-reads A through L1 (2,003 refined n = 100 systems 3.65 ms, 4.68 with the
    // widest split).
    k.widest_smem = FAM != FAM_CUBIC;
    k.per_cta = 1;
    return k;
}

} // namespace nls
