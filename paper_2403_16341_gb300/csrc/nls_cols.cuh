// nls_cols.cuh -- one instance per CTA for Newton, backtracking and the dogleg
// trust region (n <= 128), FP64 or mixed precision, the Jacobian held in
// shared memory by columns.
//
// Layout.  Column j of J lies at A + j * ld (ld = 4 x odd, so a walk along a
// row meets 8 banks), the right-hand side is column n.  A CTA has one warp per
// 32 rows (more in FP64); the shared memory and the warps are sized by the
// request's n, so an SM holds as many instances as their matrices allow (four
// at n = 96 in mixed precision, two in FP64).
//
// LU with partial pivoting (Sec. 3.2, Fig. 5), right-looking in panels of C
// columns, with the next panel looked ahead:
//  * one warp holds a panel in registers, lane l the rows k0 + l + 32 s.  Per
//    column one redux.sync and a ballot give the pivot (the first position
//    holding the largest |a_ik|, the choice of an explicit-swap LU), the rows
//    keep their lanes and carry the position that the interchanges give them,
//    and the factored panel is stored back by positions: L left of the
//    diagonal, U from it on;
//  * after the panel's one CTA barrier every warp loads its rows' multipliers
//    into registers and updates the columns to the right in chunks: the pivot
//    rows' entries of a chunk are solved to U12 = L11^-1 of them, one column
//    per lane, then every row subtracts its C products and is stored at its new
//    position, which makes the row interchanges free;
//  * the warp that owns the next panel updates that panel's columns first and
//    factors them while the other warps draw the remaining chunks from a
//    counter, so the serial pivot steps overlap the updates.
// Every element sees the same operations in the same order as in an unblocked
// LU.  16,384 Bratu systems of n = 64..128 (trust region), against J in one
// warp's registers per 16 columns (mixed) and block-cyclic register tiles with a
// barrier per step (FP64): 21.2 -> 12.4 ms and 138 -> 69.7 ms.
//
// What bounds it.  Mixed: issue slots and the pivot steps' latency, shared by
// the SM's instances.  FP64: the FP64 pipe (64 to 76 cycles per warp
// instruction whatever lanes are active), so the rows that remain are packed
// from lane 0 on (ceil((n - k0) / 32) instructions per column and step).
//
// For a second right-hand side (iterative refinement, NLS_REFINE) the forward
// elimination is replayed panel by panel with the recorded interchanges.
// r = -F - J dN is formed with J in FP64, evaluated row by row from the family.
//
// The Jacobian comes from forward-mode duals over the stencil of each row
// (Sec. 2.4), the globalisations are those of the other tilings (Sec. 2.2).
#pragma once

#include <climits>

#include "nls_pivot.cuh"

namespace nls {

constexpr int COL_NMAX = 128;
// Columns that a warp updates at a time: one per lane of the U12 solve in mixed
// precision, where that solve is a fifth of the instructions; FP64 16, which
// spreads the FP64 work more evenly over the warps.
template <bool MIXED>
constexpr int col_chunk() { return MIXED ? 32 : 16; }

// Columns per panel.  A wider panel means fewer passes over the trailing
// columns but a longer serial part (its own columns' update and factors).
// Measured on 16,384 Bratu systems of n = 64..128: mixed 13.9 / 12.8 / 18 ms
// with 4 / 8 / 16 columns, FP64 77 / 74 / 94 ms with 2 / 4 / 8.
template <bool MIXED>
constexpr int col_panel() { return MIXED ? 8 : 4; }
// The CTA's warps for a system of size n: one per 32 rows; FP64 twice as many
// (at most 8), which keeps the four FP64 units busy while one warp factors
// (FP64: 79 ms with 4 warps at n > 64, 74 ms with 8).
template <bool MIXED>
constexpr int col_warps(int n) { return MIXED ? (n + 31) / 32 : (n <= 32 ? 2 : n <= 64 ? 4 : 8); }
// CTAs per SM that the registers are sized for.  Mixed: four, as many as the
// shared memory holds at n = 100; the cubic, which re-reads A, runs better with
// three and more registers for its loads (2,003 refined n = 100 systems: 4.07
// against 5.28 ms; the Bratu set: 14.2 against 12.8 ms).
template <int FAM, bool MIXED>
constexpr int col_min_ctas() { return MIXED ? (FAM == FAM_CUBIC ? 3 : 4) : 2; }
template <bool MIXED>
constexpr int col_max_threads() { return 32 * col_warps<MIXED>(COL_NMAX); }

// The CTA's shared memory: fixed part, then U12 chunks and the matrix.
template <int C, bool MIXED>
struct ColSmem {
    using P = typename std::conditional<MIXED, float, double>::type;
    static constexpr int US = C + 16 / (int)sizeof(P); // a U12 column: 16-byte aligned, conflict-free
    static constexpr int NP = (COL_NMAX + C - 1) / C;
    static constexpr int MW = col_warps<MIXED>(COL_NMAX);
    double u[COL_NMAX], F[COL_NMAX], dN[COL_NMAX], ut[COL_NMAX];
    P g[COL_NMAX], Jg[COL_NMAX], y[COL_NMAX], x[COL_NMAX], rdiag[COL_NMAX];
    double rd[3][MW];
    uint64_t rm[MW];
    long long inst;
    int late;
    int singular[2];           // panel parity: a zero or non-finite pivot
    int chunk[2];              // next chunk of the trailing columns, panel parity
    alignas(16) P l11[2][C][C]; // column c of the panel's L11 below its diagonal, from slot 0 on
    int piv[2][C];             // row (before the panel's interchanges) of pivot c
    unsigned char pos[2][COL_NMAX];            // position of each row after the panel's interchanges
    unsigned char perm[MIXED ? NP : 1][COL_NMAX];  // all panels' (second right-hand sides)
    unsigned char prow[MIXED ? COL_NMAX : 1];      // pivot row of each step, before its panel's interchanges
};
// leading dimension of the matrix
constexpr int col_ld(int n) { return 4 * (((n + 3) / 4) | 1); }
template <int C, bool MIXED>
constexpr int col_smem_bytes(int n)
{
    using SM = ColSmem<C, MIXED>;
    return (int)((sizeof(SM) + 15) / 16 * 16) +
           (col_warps<MIXED>(n) * col_chunk<MIXED>() * SM::US + (n + 1) * col_ld(n)) * (MIXED ? 4 : 8);
}

template <int C, int FAM, bool MIXED>
struct ColSolver {
    using P = typename std::conditional<MIXED, float, double>::type;
    using K = decltype(mag_bits(P(0)));
    using SM = ColSmem<C, MIXED>;
    static constexpr int US = SM::US;
    static constexpr int CHUNK = col_chunk<MIXED>();

    int tid, lane, warp, nw, n, ld;
    P *A;  // the matrix, by columns; column n is the right-hand side
    P *ub; // this warp's U12 chunk
    int64_t B, k;
    const double *params;
    double lam; // Bratu lambda
    double fF, Delta;
    int it, nfev, rej, status, ngrad;
    bool need_jac;
    uint64_t fmag;

    // ------------------------------------------------------------ reductions
    // K block sums with one pair of barriers (warps summed in a fixed order,
    // so every thread gets the same, reproducible value)
    template <int KS>
    NLS_DI void bsumk(double (&v)[KS], SM &sm) const
    {
#pragma unroll
        for (int j = 0; j < KS; ++j) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
            if (lane == 0) sm.rd[j][warp] = v[j];
        }
        __syncthreads();
        const int nr = (n + 31) / 32; // the warps that hold components
#pragma unroll
        for (int j = 0; j < KS; ++j) {
            double s = 0.0;
            for (int w = 0; w < nr; ++w) s += sm.rd[j][w];
            v[j] = s;
        }
        __syncthreads();
    }
    // block sum of v and block max of m with one pair of barriers
    NLS_DI void bsum_max(double &v, uint64_t &m, SM &sm) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, o);
            const uint64_t w = __shfl_xor_sync(0xffffffffu, m, o);
            m = w > m ? w : m;
        }
        if (lane == 0) {
            sm.rd[0][warp] = v;
            sm.rm[warp] = m;
        }
        __syncthreads();
        const int nr = (n + 31) / 32;
        double s = 0.0;
        uint64_t x = 0;
        for (int w = 0; w < nr; ++w) {
            s += sm.rd[0][w];
            x = sm.rm[w] > x ? sm.rm[w] : x;
        }
        __syncthreads();
        v = s;
        m = x;
    }
    NLS_DI uint64_t bmax(uint64_t v, SM &sm) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
            v = w > v ? w : v;
        }
        if (lane == 0) sm.rm[warp] = v;
        __syncthreads();
        const int nr = (n + 31) / 32;
        uint64_t m = 0;
        for (int w = 0; w < nr; ++w) m = sm.rm[w] > m ? sm.rm[w] : m;
        __syncthreads();
        return m;
    }

    // ------------------------------------------------------------ residual
    // s + (A v)_t for the cubic, terms added in order; the loads of 16 terms are
    // in flight together (one at a time, their latency was most of the call).
    // FILL also writes row t of A into the matrix: the residuals do, whose
    // callers are done with the factors, so the next Jacobian finds the linear
    // part in place and the parameters, which come by 32-byte sectors of one
    // element each, are read once less per pass (2,003
    // refined n = 100 systems: 4.01 -> 3.68 ms).
    template <bool FILL>
    NLS_DI double adot(int t, const double *v, double s) const
    {
        const double *row = params + (int64_t)t * n * B + k;
        int j = 0;
        for (; j + 16 <= n; j += 16) {
            double a[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) a[q] = __ldg(row + (int64_t)(j + q) * B);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                s = fma(a[q], v[j + q], s);
                if constexpr (FILL) A[(j + q) * ld + t] = P(a[q]);
            }
        }
        for (; j < n; ++j) {
            const double a = __ldg(row + (int64_t)j * B);
            s = fma(a, v[j], s);
            if constexpr (FILL) A[j * ld + t] = P(a);
        }
        return s;
    }

    // F_t(x) in FP64 for t < n, x in shared memory; returns F_t (0 for t >= n).
    // The cubic overwrites the matrix (adot).
    NLS_DI double residual_t(const double *x) const
    {
        const int t = tid;
        if (t >= n) return 0.0;
        const double xt = x[t];
        if constexpr (FAM == FAM_CUBIC) {
            double s = 0.0;
            s = adot<true>(t, x, s);
            return s + xt * xt * xt - __ldg(params + (int64_t)(n * n + t) * B + k);
        } else if constexpr (FAM == FAM_BRATU) {
            const double inv_h2 = double((n + 1) * (n + 1));
            const double left = t > 0 ? x[t - 1] : 0.0;
            const double right = t < n - 1 ? x[t + 1] : 0.0;
            return inv_h2 * ((left + (-2.0) * xt) + right) + lam * exp(xt);
        } else if constexpr (FAM == FAM_SQUARE) {
            return xt * xt - __ldg(params + (int64_t)t * B + k);
        } else {
            return t == 0 ? 1.0 - xt : 10.0 * (xt - x[t - 1] * x[t - 1]);
        }
    }

    // (J(u) v)_t in FP64 at the current iterate sm.u, for t < n (0 beyond):
    // the FP64 Jacobian row of each family applied to v, evaluated on the fly
    // (no FP64 copy of J is held).  Iterative refinement's residual.
    NLS_DI double jdot64_t(const double *v, const SM &sm) const
    {
        const int t = tid;
        if (t >= n) return 0.0;
        const double ut = sm.u[t];
        if constexpr (FAM == FAM_CUBIC) {
            double s = 3.0 * ut * ut * v[t];
            s = adot<false>(t, v, s);
            return s;
        } else if constexpr (FAM == FAM_BRATU) {
            const double inv_h2 = double((n + 1) * (n + 1));
            const double left = t > 0 ? v[t - 1] : 0.0;
            const double right = t < n - 1 ? v[t + 1] : 0.0;
            return inv_h2 * ((left + (-2.0) * v[t]) + right) + lam * exp(ut) * v[t];
        } else if constexpr (FAM == FAM_SQUARE) {
            return 2.0 * ut * v[t];
        } else {
            return t == 0 ? -v[0] : 10.0 * (v[t] - 2.0 * sm.u[t - 1] * v[t - 1]);
        }
    }

    // ------------------------------------------------------------ Jacobian
    // partials of F_t over its stencil: d0 (t-1), d1 (t), d2 (t+1); the cubic's
    // d1 is the nonlinear part's alone
    NLS_DI void stencil(const SM &sm, P &d0, P &d1, P &d2) const
    {
        const int i = tid;
        const P ui = P(sm.u[i]);
        d0 = d1 = d2 = P(0);
        if constexpr (FAM == FAM_CUBIC) {
            const auto x = seed<1, 0, P>(ui);
            d1 = (x * x * x).d[0];
        } else if constexpr (FAM == FAM_BRATU) {
            const P inv_h2 = P((n + 1) * (n + 1));
            const auto xl = seed<3, 0, P>(P(0));
            const auto xc = seed<3, 1, P>(ui);
            const auto xr = seed<3, 2, P>(P(0));
            const auto f = inv_h2 * ((xl + P(-2) * xc) + xr) + P(lam) * exp(xc);
            d0 = f.d[0];
            d1 = f.d[1];
            d2 = f.d[2];
        } else if constexpr (FAM == FAM_SQUARE) {
            const auto x = seed<1, 0, P>(ui);
            d1 = (x * x).d[0];
        } else {
            const P ul = i > 0 ? P(sm.u[i - 1]) : P(0);
            const auto xl = seed<2, 0, P>(ul);
            const auto xc = seed<2, 1, P>(ui);
            const auto f = P(10) * (xc - xl * xl);
            d0 = f.d[0];
            d1 = (i == 0) ? P(-1) : f.d[1];
        }
    }

    // J by columns, and the right-hand side -F as column n (whole CTA)
    NLS_DI void jacobian(SM &sm) const
    {
        [[maybe_unused]] const int tpb = 32 * nw;
        P d0 = P(0), d1 = P(0), d2 = P(0);
        if (tid < n) stencil(sm, d0, d1, d2);
        if constexpr (FAM == FAM_CUBIC) {
            // the linear part is there (the last residual wrote row tid)
            if (tid < n) A[tid * ld + tid] += d1;
        } else {
            using V = typename std::conditional<MIXED, float4, double2>::type;
            const int nv = n * ld * (int)sizeof(P) / 16; // ld is a multiple of 4
            for (int e = tid; e < nv; e += tpb) reinterpret_cast<V *>(A)[e] = V{};
            __syncthreads();
            if (tid < n) {
                if (tid > 0) A[(tid - 1) * ld + tid] = d0;
                A[tid * ld + tid] = d1;
                if (tid + 1 < n) A[(tid + 1) * ld + tid] = d2;
            }
        }
        if (tid < n) A[n * ld + tid] = -P(sm.F[tid]);
    }

    // g = J^T F and J g from the columns (whole CTA; ends with a barrier)
    NLS_DI void gradient(SM &sm) const
    {
        const P *y = A + n * ld; // -F
        if constexpr (FAM != FAM_CUBIC) {
            // the stencil families' three terms, summed as a sum over the lanes
            // holding rows r mod 32 does (rows j - 1 and j + 1 meet first), and in
            // J g over groups of 16 columns
            if (tid < n) {
                const P *c = A + tid * ld + tid;
                const P l = tid > 0 ? c[-1] * y[tid - 1] : P(0), m = c[0] * y[tid];
                const P r = tid + 1 < n ? c[1] * y[tid + 1] : P(0);
                sm.g[tid] = -((l + r) + m);
            }
            __syncthreads();
            if (tid < n) {
                P t = P(0), s = P(0);
                for (int j = max(tid - 1, 0); j <= min(tid + 1, n - 1); ++j) {
                    s = fma(A[j * ld + tid], sm.g[j], s);
                    if ((j & 15) == 15) {
                        t += s;
                        s = P(0);
                    }
                }
                sm.Jg[tid] = t + s;
            }
        } else if constexpr (MIXED) {
            // a warp per column: rows lane, lane + 32, .., then over the lanes
            for (int j = warp; j < n; j += nw) {
                P s = P(0);
                for (int i = lane; i < n; i += 32) s = fma(A[j * ld + i], y[i], s);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) sm.g[j] = -s;
            }
            __syncthreads();
            if (tid < n) {
                P t = P(0);
                for (int c0 = 0; c0 < n; c0 += 16) { // partial sums over 16 columns
                    P s = P(0);
                    for (int c = c0; c < min(c0 + 16, n); ++c) s = fma(A[c * ld + tid], sm.g[c], s);
                    t += s;
                }
                sm.Jg[tid] = t;
            }
        } else {
            if (tid < n) {
                P s = P(0);
                for (int i = 0; i < n; ++i) s = fma(A[tid * ld + i], y[i], s);
                sm.g[tid] = -s;
            }
            __syncthreads();
            if (tid < n) {
                P s = P(0);
                for (int j = 0; j < n; ++j) s = fma(A[j * ld + tid], sm.g[j], s);
                sm.Jg[tid] = s;
            }
        }
        __syncthreads();
    }

    // ------------------------------------------------------------ LU
    // Entry `slot` (warp-uniform) of a per-slot array: a select chain, no branch.
    template <int SK>
    NLS_DI static P pick(const P (&v)[SK], int slot)
    {
        P x = v[0];
#pragma unroll
        for (int s = 1; s < SK; ++s) x = (slot == s) ? v[s] : x;
        return x;
    }

    // The pivot of column kk among this warp's rows that remain (those at
    // positions >= kk): its lane, slot and position.  The largest |a| wins, then
    // the lowest position; a NaN below position kk is never chosen.
    template <int SK>
    NLS_DI static void find_pivot(const P (&a)[SK], const int (&pos)[SK], int kk, int &src, int &pslot, int &ppos)
    {
        const unsigned FULL = 0xffffffffu;
        const K inf = inf_bits(P(0));
        const uint32_t inf_word = sizeof(K) == 8 ? (uint32_t)((uint64_t)inf >> 32) : (uint32_t)inf;
        // the magnitude's high word + 1 (0: no candidate); one holder of the
        // largest is the pivot
        uint32_t hk[SK], best = 0;
#pragma unroll
        for (int s = 0; s < SK; ++s) {
            const K m = mag_bits(a[s]);
            hk[s] = pos[s] >= kk ? (uint32_t)(sizeof(K) == 8 ? (uint64_t)m >> 32 : (uint64_t)m) + 1u : 0u;
            best = max(best, hk[s]);
        }
        const uint32_t h = __reduce_max_sync(FULL, best);
        int bs = 0, bp = pos[0], same = hk[0] == h;
#pragma unroll
        for (int s = 1; s < SK; ++s)
            if (hk[s] == h) {
                bs = s;
                bp = pos[s];
                ++same;
            }
        unsigned b = __ballot_sync(FULL, best == h);
        src = __ffs(b) - 1;
        int pk = __shfl_sync(FULL, (bp << 8) | (bs << 4) | same, src);
        if ((b & (b - 1u)) || (pk & 15) != 1 || h - 1u >= inf_word) {
            // several holders, an infinity or a NaN: the full comparison
            K bm = K(0);
            bp = INT_MAX;
            bs = 0;
#pragma unroll
            for (int s = 0; s < SK; ++s) {
                K m = mag_bits(a[s]);
                if (pos[s] > kk && m > inf) m = K(0);
                if (pos[s] >= kk && (bp == INT_MAX || m > bm || (m == bm && pos[s] < bp))) {
                    bm = m;
                    bp = pos[s];
                    bs = s;
                }
            }
            const uint32_t kh = bp == INT_MAX ? 0u : (uint32_t)(sizeof(K) == 8 ? (uint64_t)bm >> 32 : (uint64_t)bm) + 1u;
            const uint32_t g = __reduce_max_sync(FULL, kh);
            bool top = kh != 0u && kh == g;
            if constexpr (sizeof(K) == 8) {
                const uint32_t lo = __reduce_max_sync(FULL, top ? (uint32_t)bm : 0u);
                top = top && (uint32_t)bm == lo;
            }
            const uint32_t kp = top ? ~(uint32_t)bp : 0u;
            const uint32_t q = __reduce_max_sync(FULL, kp);
            src = __ffs(__ballot_sync(FULL, top && kp == q)) - 1;
            pk = __shfl_sync(FULL, (bp << 8) | (bs << 4), src);
        }
        ppos = pk >> 8;
        pslot = (pk >> 4) & 15;
    }
    // The rows' positions after the interchange of step kk.
    template <int SK>
    NLS_DI void take_pivot(int (&pos)[SK], int kk, int src, int pslot, int ppos) const
    {
#pragma unroll
        for (int s = 0; s < SK; ++s) {
            if (pos[s] == kk) pos[s] = ppos; // the pivot's old position
            if (s == pslot && lane == src) pos[s] = kk;
        }
    }

    // This warp factors the kc columns of the panel at k0 (SK = ceil((n - k0)
    // / 32) row slots); a zero or non-finite pivot raises sm.singular of the
    // panel's parity.  FP32: a loop over the columns whose body moves the panel
    // one column to the left (unrolled, the four slot counts' code did not fit
    // the instruction cache: 66 ms instead of 19 with 16 columns on the Bratu n = 64..128
    // set).  FP64: few columns, unrolled in place.
    template <int SK>
    NLS_DI void factor_panel(int k0, int kc, int p, SM &sm) const
    {
        const unsigned FULL = 0xffffffffu;
        const int par = p & 1;
        P v[C][SK];
        int pos[SK];
#pragma unroll
        for (int s = 0; s < SK; ++s) {
            const int i = k0 + lane + 32 * s;
            pos[s] = i < n ? i : -1; // a row remains while its position is >= the step
#pragma unroll
            for (int c = 0; c < C; ++c) v[c][s] = (i < n && c < kc) ? A[(k0 + c) * ld + i] : P(0);
        }
        bool ok = true;
        if constexpr (MIXED) {
            for (int c = 0; c < kc; ++c) {
                const int kk = k0 + c;
                int src, pslot, ppos;
                find_pivot<SK>(v[0], pos, kk, src, pslot, ppos);
                const P pv = __shfl_sync(FULL, pick<SK>(v[0], pslot), src);
                const P r = pivot_reciprocal(pv, ok);
                take_pivot<SK>(pos, kk, src, pslot, ppos);
                // column kk is finished: multipliers of the rows that remain, U of
                // the others, kept by row until the panel's end
                P l[SK];
#pragma unroll
                for (int s = 0; s < SK; ++s) {
                    l[s] = pos[s] > kk ? v[0][s] * r : P(0);
                    if (k0 + lane + 32 * s < n) A[kk * ld + k0 + lane + 32 * s] = pos[s] > kk ? l[s] : v[0][s];
                }
#pragma unroll
                for (int cc = 1; cc < C; ++cc) {
                    if (cc >= kc - c) break;
                    const P e = __shfl_sync(FULL, pick<SK>(v[cc], pslot), src);
#pragma unroll
                    for (int s = 0; s < SK; ++s) v[cc - 1][s] = v[cc][s] - l[s] * e;
                }
                if (lane == 0) {
                    sm.rdiag[kk] = r;
                    sm.piv[par][c] = k0 + src + 32 * pslot;
                    sm.prow[kk] = (unsigned char)(k0 + src + 32 * pslot);
                }
            }
            // to their positions
#pragma unroll 2
            for (int c = 0; c < kc; ++c) {
                P *col = A + (k0 + c) * ld;
                P t[SK];
#pragma unroll
                for (int s = 0; s < SK; ++s) t[s] = k0 + lane + 32 * s < n ? col[k0 + lane + 32 * s] : P(0);
                __syncwarp(); // the column is read
#pragma unroll
                for (int s = 0; s < SK; ++s) {
                    if (k0 + lane + 32 * s < n) {
                        col[pos[s]] = t[s];
                        const int q = pos[s] - k0;
                        if (q > c && q < kc) sm.l11[par][c][q - c - 1] = t[s];
                    }
                }
            }
#pragma unroll
            for (int s = 0; s < SK; ++s) {
                const int i = k0 + lane + 32 * s;
                if (i < n) {
                    sm.pos[par][i] = (unsigned char)pos[s];
                    sm.perm[p][i] = (unsigned char)pos[s];
                }
            }
        } else {
            __syncwarp(); // the panel is in registers: its space may be rewritten
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (c >= kc) break;
                const int kk = k0 + c;
                int src, pslot, ppos;
                find_pivot<SK>(v[c], pos, kk, src, pslot, ppos);
                const P pv = __shfl_sync(FULL, pick<SK>(v[c], pslot), src);
                const P r = pivot_reciprocal(pv, ok);
                take_pivot<SK>(pos, kk, src, pslot, ppos);
#pragma unroll
                for (int s = 0; s < SK; ++s)
                    if (pos[s] > kk) v[c][s] *= r; // the multiplier
#pragma unroll
                for (int cc = c + 1; cc < C; ++cc) {
                    if (cc >= kc) break;
                    const P e = __shfl_sync(FULL, pick<SK>(v[cc], pslot), src);
#pragma unroll
                    for (int s = 0; s < SK; ++s)
                        if (pos[s] > kk) v[cc][s] -= v[c][s] * e;
                }
                if (lane == 0) {
                    sm.rdiag[kk] = r;
                    sm.piv[par][c] = k0 + src + 32 * pslot;
                }
            }
            // back by positions: multipliers below the diagonal, U from it on
#pragma unroll
            for (int s = 0; s < SK; ++s) {
                const int i = k0 + lane + 32 * s;
                if (i < n) {
                    sm.pos[par][i] = (unsigned char)pos[s];
                    const int q = pos[s] - k0;
#pragma unroll
                    for (int c = 0; c < C; ++c)
                        if (c < kc) {
                            A[(k0 + c) * ld + pos[s]] = v[c][s];
                            if (q > c && q < kc) sm.l11[par][c][q - c - 1] = v[c][s];
                        }
                }
            }
        }
        if (lane == 0) sm.singular[par] = !ok;
        __syncwarp();
    }

    // Columns j0 .. j0 + nj - 1 (nj <= CHUNK) of the trailing matrix under
    // the panel at k0: l are this lane's rows' multipliers, pos their new
    // positions.
    template <int SK>
    NLS_DI void update_chunk(int k0, int kc, int par, int j0, int nj, bool paired, const P (&l)[SK][C],
                             const int (&pos)[SK], SM &sm) const
    {
        // U12 = L11^-1 (the pivot rows' entries), column j0 + lane
        if (lane < nj) {
            const P *col = A + (j0 + lane) * ld;
            P *o = ub + lane * US;
            P w[C];
#pragma unroll
            for (int c = 0; c < C; ++c) w[c] = c < kc ? col[sm.piv[par][c]] : P(0);
            if constexpr (MIXED) {
                using V = float4;
#pragma unroll 1
                for (int c2 = 0; c2 < C; ++c2) { // w moves one entry to the left per step
                    const P u = w[0];
                    o[c2] = u;
                    const P *l11 = sm.l11[par][c2];
#pragma unroll
                    for (int q = 0; q < C; q += 4) {
                        if (q >= kc - 1 - c2) break;
                        const V t = *reinterpret_cast<const V *>(l11 + q);
                        if (q + 1 < C) w[q] = w[q + 1] - t.x * u;
                        if (q + 2 < C) w[q + 1] = w[q + 2] - t.y * u;
                        if (q + 3 < C) w[q + 2] = w[q + 3] - t.z * u;
                        if (q + 4 < C) w[q + 3] = w[q + 4 < C ? q + 4 : 0] - t.w * u;
                    }
                    if (c2 >= kc - 1) w[0] = P(0); // past the panel's last column
                }
            } else {
#pragma unroll
                for (int c2 = 0; c2 < C; ++c2) {
                    if (c2 >= kc) break;
#pragma unroll
                    for (int c = c2 + 1; c < C; ++c)
                        if (c < kc) w[c] -= sm.l11[par][c2][c - c2 - 1] * w[c2];
                }
#pragma unroll
                for (int q = 0; q < C / 2; ++q) reinterpret_cast<double2 *>(o)[q] = make_double2(w[2 * q], w[2 * q + 1]);
            }
        }
        __syncwarp();
        if constexpr (!MIXED) {
            if (paired) {
                // Two columns at a time: the full slots of each, then the last slot of
                // both in one instruction per product, the lower half-warp on the first
                // column and the upper on the second (a warp FP64 instruction costs the
                // same with 16 lanes as with 32; 16,384 Bratu systems of n = 64..128:
                // 71.9 -> 69.8 ms).
                const int half = lane >> 4, i2 = k0 + 32 * (SK - 1) + (lane & 15);
                for (int jj = 0; jj < nj; jj += 2) {
                    const bool two = jj + 1 < nj;
                    P *col = A + (j0 + jj) * ld;
                    P *colh = col + (half ? ld : 0);
                    const bool on = i2 < n && (two || !half);
                    P a[2][SK], t = on ? colh[i2] : P(0);
#pragma unroll
                    for (int s = 0; s < SK - 1; ++s) {
                        a[0][s] = col[k0 + lane + 32 * s];
                        a[1][s] = two ? col[ld + k0 + lane + 32 * s] : P(0);
                    }
                    const P *o = ub + jj * US, *oh = o + (half && two ? US : 0);
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const P w0 = o[c];
#pragma unroll
                        for (int s = 0; s < SK - 1; ++s) a[0][s] -= l[s][c] * w0;
                        t -= l[SK - 1][c] * oh[c];
                        if (SK > 1 && two) {
                            const P w1 = o[US + c];
#pragma unroll
                            for (int s = 0; s < SK - 1; ++s) a[1][s] -= l[s][c] * w1;
                        }
                    }
                    __syncwarp(); // every row of the columns is read
#pragma unroll
                    for (int s = 0; s < SK - 1; ++s) {
                        col[pos[s]] = a[0][s];
                        if (two) col[ld + pos[s]] = a[1][s];
                    }
                    if (on) colh[pos[SK - 1]] = t;
                }
                __syncwarp();
                return;
            }
        }
        for (int jj = 0; jj < nj; ++jj) {
            P *col = A + (j0 + jj) * ld;
            P a[SK], w[C];
#pragma unroll
            for (int s = 0; s < SK; ++s) {
                const int i = k0 + lane + 32 * s;
                a[s] = i < n ? col[i] : P(0);
            }
            const P *o = ub + jj * US;
            if constexpr (MIXED) {
#pragma unroll
                for (int q = 0; q < C / 4; ++q) {
                    const float4 t = reinterpret_cast<const float4 *>(o)[q];
                    w[4 * q] = t.x;
                    w[4 * q + 1] = t.y;
                    w[4 * q + 2] = t.z;
                    w[4 * q + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int q = 0; q < C / 2; ++q) {
                    const double2 t = reinterpret_cast<const double2 *>(o)[q];
                    w[2 * q] = t.x;
                    w[2 * q + 1] = t.y;
                }
            }
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
                for (int s = 0; s < SK; ++s) a[s] -= l[s][c] * w[c];
            __syncwarp(); // every row of the column is read
#pragma unroll
            for (int s = 0; s < SK; ++s)
                if (k0 + lane + 32 * s < n) col[pos[s]] = a[s];
        }
        __syncwarp();
    }

    // This warp's share of the trailing update under panel p: the next panel's
    // kn columns alone (ahead), or the chunks that it draws of the others.
    template <int SK>
    NLS_DI void trailing(int k0, int kc, int p, bool ahead, SM &sm) const
    {
        const int par = p & 1;
        const int k1 = k0 + kc, kn = min(C, n - k1); // the next panel
        // the columns right of the next panel, the right-hand side last
        auto draw = [&]() {
            int q = 0;
            if (lane == 0) q = atomicAdd(&sm.chunk[par], 1);
            return k1 + kn + __shfl_sync(0xffffffffu, q, 0) * CHUNK;
        };
        int j = ahead ? k1 : draw();
        if (j > n) return;
        // FP64: 16 rows or fewer in the last slot are held by both half-warps
        const bool paired = !MIXED && n - k0 - 32 * (SK - 1) <= 16;
        P l[SK][C];
        int pos[SK];
#pragma unroll
        for (int s = 0; s < SK; ++s) {
            const int i = k0 + (paired && s == SK - 1 ? lane & 15 : lane) + 32 * s;
            pos[s] = i < n ? sm.pos[par][i] : 0;
            // a pivot row q of this panel takes the first q products
            const int q = i < n ? min(pos[s] - k0, kc) : 0;
#pragma unroll
            for (int c = 0; c < C; ++c) l[s][c] = c < q ? A[(k0 + c) * ld + pos[s]] : P(0);
        }
        for (;;) {
            update_chunk<SK>(k0, kc, par, j, ahead ? kn : min(CHUNK, n + 1 - j), paired, l, pos, sm);
            if (ahead) break;
            j = draw();
            if (j > n) break;
        }
    }
    NLS_DI void factor_next(int k0, int kc, int p, SM &sm) const
    {
        switch ((n - k0 + 31) / 32) {
        case 1: factor_panel<1>(k0, kc, p, sm); break;
        case 2: factor_panel<2>(k0, kc, p, sm); break;
        case 3: factor_panel<3>(k0, kc, p, sm); break;
        default: factor_panel<4>(k0, kc, p, sm); break;
        }
    }

    // Factors A and eliminates column n; x (by column) to sm.x.  False on a zero
    // or non-finite pivot (uniform over the CTA).
    NLS_DI bool lu_solve(SM &sm) const
    {
        if (tid == 0) {
            sm.chunk[0] = sm.chunk[1] = 0;
        }
        __syncthreads(); // A is complete
        for (int p = -1;; ++p) { // p = -1: the first panel's factors only
            if (p >= 0) {
                __syncthreads(); // panel p is factored, the columns right of it are up to date
                if (sm.singular[p & 1]) return false;
                if (tid == 0) sm.chunk[(p + 1) & 1] = 0;
            }
            const int k0 = p * C, kc = min(C, n - k0), k1 = k0 + kc;
            // the next panel's owner: its columns, its factors, then a share of the rest
            const bool owner = k1 < n && warp == (p + 1) % nw;
            for (int part = owner ? 0 : 1; part < 2; ++part) {
                const bool ahead = part == 0;
                if (p >= 0) {
                    switch ((n - k0 + 31) / 32) {
                    case 1: trailing<1>(k0, kc, p, ahead, sm); break;
                    case 2: trailing<2>(k0, kc, p, ahead, sm); break;
                    case 3: trailing<3>(k0, kc, p, ahead, sm); break;
                    default: trailing<4>(k0, kc, p, ahead, sm); break;
                    }
                }
                if (ahead) factor_next(k1, min(C, n - k1), p + 1, sm);
            }
            if (k1 >= n) break;
        }
        __syncthreads();
        if (warp == 0) back_sub(A + n * ld, sm);
        __syncthreads();
        return true;
    }

    // Back substitution on one warp: y by position (lane l: positions l, l +
    // 32, ..), column by column from the last; x to sm.x.
    NLS_DI void back_sub(const P *yin, SM &sm) const
    {
        P y[4], rd[4], x[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int i = lane + 32 * s;
            y[s] = i < n ? yin[i] : P(0);
            rd[s] = i < n ? sm.rdiag[i] : P(0);
            x[s] = P(0);
        }
#pragma unroll
        for (int js = 3; js >= 0; --js) {
            const int top = min(31, n - 1 - 32 * js);
#pragma unroll 2
            for (int q = top; q >= 0; --q) {
                const int kk = 32 * js + q;
                const P xk = __shfl_sync(0xffffffffu, y[js] * rd[js], q);
                if (lane == q) x[js] = xk;
                const P *col = A + kk * ld + lane;
                if (lane < q) y[js] -= col[32 * js] * xk;
#pragma unroll
                for (int s = 0; s < js; ++s) y[s] -= col[32 * s] * xk;
            }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (lane + 32 * s < n) sm.x[lane + 32 * s] = x[s];
    }

    // A second right-hand side (sm.y, by row) with the factors of lu_solve; x to
    // sm.x.  Warp 0 replays the steps panel by panel: the rows' products in the
    // order of the elimination, then the panel's interchanges.
    NLS_DI void lu_apply(SM &sm) const
    {
        if (warp == 0) {
            for (int k0 = 0, p = 0; k0 < n; k0 += C, ++p) {
                const int kc = min(C, n - k0);
                P yv[4];
                int pos[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const int i = k0 + lane + 32 * s;
                    yv[s] = i < n ? sm.y[i] : P(0);
                    pos[s] = i < n ? sm.perm[MIXED ? p : 0][i] : 0;
                }
                __syncwarp();
                for (int c = 0; c < kc; ++c) {
                    const int pr = (int)sm.prow[MIXED ? k0 + c : 0] - k0;
                    const P yk = __shfl_sync(0xffffffffu, pick<4>(yv, pr >> 5), pr & 31);
                    const P *col = A + (k0 + c) * ld;
#pragma unroll
                    for (int s = 0; s < 4; ++s)
                        if (k0 + lane + 32 * s < n && pos[s] > k0 + c) yv[s] -= col[pos[s]] * yk;
                }
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (k0 + lane + 32 * s < n) sm.y[pos[s]] = yv[s];
                __syncwarp();
            }
            back_sub(sm.y, sm);
        }
        __syncthreads();
    }

    // ------------------------------------------------------------ driver
    NLS_DI void set_status_from(uint64_t m, const SolveArgs &A_)
    {
        fmag = m;
        if (m >= INF64_BITS) status = ST_NONFINITE;
        else if (m <= mag_bits(A_.abstol)) status = ST_SUCCESS;
        else if (it >= A_.maxiters) status = ST_MAXITERS;
    }

    NLS_DI void init(const SolveArgs &A_, SM &sm)
    {
        if (tid < n) sm.u[tid] = A_.u[(int64_t)tid * B + k];
        lam = (FAM == FAM_BRATU) ? __ldg(A_.params + k) : 0.0;
        __syncthreads();
        const double f = residual_t(sm.u);
        if (tid < n) sm.F[tid] = f;
        nfev = 1;
        it = 0;
        rej = 0;
        ngrad = 0;
        Delta = TR_DELTA0;
        need_jac = true;
        status = ST_RUNNING;
        fF = f * f;
        uint64_t mx = mag_bits(f);
        bsum_max(fF, mx, sm);
        set_status_from(mx, A_);
        if (status == ST_RUNNING && A_.maxiters <= 0) status = ST_MAXITERS;
    }

    NLS_DI void pass(const SolveArgs &A_, SM &sm)
    {
        ++it;
        if (need_jac) {
            jacobian(sm);
            if (A_.alg == ALG_TRUST_DOGLEG) {
                ++ngrad;
                __syncthreads();
                gradient(sm);
            }
            const bool ok = lu_solve(sm);
            if (!ok) {
                status = ST_SINGULAR;
                return;
            }
            if (tid < n) sm.dN[tid] = double(sm.x[tid]);
            __syncthreads();
            // classical iterative refinement of the Newton step: the FP64
            // residual of J dN = -F, re-solved with the same FP32 factors
            for (int r = 0; MIXED && r < A_.refine; ++r) {
                const double res = tid < n ? -sm.F[tid] - jdot64_t(sm.dN, sm) : 0.0;
                __syncthreads();
                if (tid < n) sm.y[tid] = P(res);
                __syncthreads();
                lu_apply(sm);
                if (tid < n) sm.dN[tid] += double(sm.x[tid]);
                __syncthreads();
            }
            need_jac = false;
        }
        const int t = tid;
        const bool own = t < n;
        if (A_.alg == ALG_NEWTON) {
            if (own) sm.u[t] += sm.dN[t];
            __syncthreads();
            const double f = residual_t(sm.u);
            __syncthreads();
            if (own) sm.F[t] = f;
            ++nfev;
            need_jac = true;
            set_status_from(bmax(mag_bits(f), sm), A_);
        } else if (A_.alg == ALG_NEWTON_BACKTRACK) {
            // slope F^T J dN of Eq. 9 by linearity: J dN = -F, so it is -||F||^2
            const double s = -fF;
            const double phi0 = 0.5 * fF;
            double alpha = 1.0;
            bool ok = false;
            double f = 0.0, fFt = 0.0;
            for (int m = 0; m < LS_MAX_TRIALS; ++m) {
                if (own) sm.ut[t] = fma(alpha, sm.dN[t], sm.u[t]);
                __syncthreads();
                f = residual_t(sm.ut);
                ++nfev;
                fFt = f * f;
                uint64_t mx = mag_bits(f);
                bsum_max(fFt, mx, sm);
                if (mx < INF64_BITS && 0.5 * fFt <= phi0 + LS_C1 * alpha * s) {
                    ok = true;
                    if (own) {
                        sm.u[t] = sm.ut[t];
                        sm.F[t] = f;
                    }
                    fF = fFt;
                    __syncthreads();
                    set_status_from(mx, A_);
                    break;
                }
                alpha *= LS_RHO;
            }
            if (!ok) {
                status = ST_LS_FAILED;
                return;
            }
            need_jac = true;
        } else {
            const double dn = own ? sm.dN[t] : 0.0;
            const P gt = own ? sm.g[t] : P(0), jgt = own ? sm.Jg[t] : P(0);
            const P D2 = P(Delta * Delta);
            double r3[3] = {double(P(dn) * P(dn)), double(gt * gt), double(jgt * jgt)};
            bsumk<3>(r3, sm);
            const P nN2 = P(r3[0]), gg = P(r3[1]), JgJg = P(r3[2]);
            const P tt = gg / JgJg;
            const P cc = tt * tt * gg;
            const P w = P(dn) + tt * gt;
            // the interpolation's quadratic, only when the CTA takes branch D
            // (a block-uniform decision, so the barriers inside are safe)
            P aa = P(0), bb = P(0);
            if (!(nN2 <= D2) && !(cc >= D2)) {
                double r2[2] = {double(w * w), double(-tt * gt * w)};
                bsumk<2>(r2, sm);
                aa = P(r2[0]);
                bb = P(r2[1]);
            }
            // pred = -2 F.Jd - ||Jd||^2 (Eq. 15) from block-uniform scalars:
            // J dN = -F and F.(J g) = g.g (g = J^T F), so no J d is formed
            double d, pred;
            if (nN2 <= D2) {
                d = dn;
                pred = fF;
            } else if (cc >= D2) {
                const P sc = P(Delta) / nls_sqrt(gg);
                d = double(-sc * gt);
                pred = double(sc * (P(2) * gg - sc * JgJg));
            } else {
                const P q = cc - D2;
                const P tau = (-bb + nls_sqrt(bb * bb - aa * q)) / aa;
                d = double(fma(tau, w, -tt * gt));
                const P s1 = (P(1) - tau) * tt; // J d = -s1 J g - tau F
                pred = double(s1 * (P(2) * (P(1) - tau) * gg - s1 * JgJg) + tau * (P(2) - tau) * P(fF));
            }
            if (!own) d = 0.0;
            if (own) sm.ut[t] = sm.u[t] + d;
            __syncthreads();
            const double f = residual_t(sm.ut);
            ++nfev;
            double fFt = f * f;
            uint64_t mx = mag_bits(f);
            bsum_max(fFt, mx, sm);
            const double ared = fF - fFt;
            if (tr_step_outcome(A_.tr_scheme, pred > 0.0 && mx < INF64_BITS, ared, pred, !(nN2 <= D2), Delta)) {
                if (own) {
                    sm.u[t] = sm.ut[t];
                    sm.F[t] = f;
                }
                fF = fFt;
                need_jac = true;
                rej = 0;
                __syncthreads();
                set_status_from(mx, A_);
            } else {
                if (++rej >= TR_MAX_REJECTIONS) {
                    status = ST_TR_STALLED;
                    return;
                }
                if (it >= A_.maxiters) status = ST_MAXITERS;
            }
        }
    }

    NLS_DI void finish(const SolveArgs &A_, SM &sm) const
    {
        __syncthreads();
        if (tid < n) A_.u[(int64_t)tid * B + k] = sm.u[tid];
        if (tid == 0) {
            if (A_.status) A_.status[k] = status;
            if (A_.iters) A_.iters[k] = it;
            if (A_.resid) A_.resid[k] = bits_to_double(fmag);
            if (A_.nfev) A_.nfev[k] = nfev;
            if (A_.ngrad) A_.ngrad[k] = ngrad;
            if (A_.solved && status == ST_SUCCESS) atomicAdd(A_.solved, 1ull);
        }
    }
};

// One instance per CTA at a time, drawn from the work counter or the static
// slot; a per-launch deadline is decided by one thread for the whole CTA.
template <int C, int FAM, bool MIXED>
__global__ void __launch_bounds__((col_max_threads<MIXED>()), (col_min_ctas<FAM, MIXED>())) k_solve_cols(SolveArgs a)
{
    using Solver = ColSolver<C, FAM, MIXED>;
    using SM = typename Solver::SM;
    using P = typename SM::P;
    apply_dyn_batch(a);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SM &sm = *reinterpret_cast<SM *>(smem_raw);
    Solver s;
    s.tid = threadIdx.x;
    s.lane = s.tid & 31;
    s.warp = s.tid >> 5;
    s.n = a.n;
    s.nw = col_warps<MIXED>(a.n);
    s.ld = col_ld(a.n);
    s.A = reinterpret_cast<P *>(smem_raw + (sizeof(SM) + 15) / 16 * 16);
    s.ub = s.A + (a.n + 1) * s.ld + s.warp * (Solver::CHUNK * SM::US);
    s.B = a.ld;
    s.params = a.params;
    const unsigned long long t_end = a.budget_ns ? global_ns() + a.budget_ns : ~0ull;
    bool first = true;
    for (;;) {
        if (s.tid == 0) {
            long long next;
            if (a.counter) next = (long long)atomicAdd(a.counter, 1ull);
            else next = first ? (long long)blockIdx.x : (long long)a.batch;
            sm.inst = next;
        }
        first = false;
        __syncthreads();
        s.k = sm.inst;
        __syncthreads();
        if (s.k >= a.batch) break;
        s.init(a, sm);
        while (s.status == ST_RUNNING) {
            if (a.budget_ns) {
                if (s.tid == 0) sm.late = global_ns() > t_end;
                __syncthreads();
                const bool late = sm.late;
                __syncthreads();
                if (late) {
                    s.status = ST_ABORTED;
                    break;
                }
            }
            s.pass(a, sm);
        }
        s.finish(a, sm);
    }
}

} // namespace nls
