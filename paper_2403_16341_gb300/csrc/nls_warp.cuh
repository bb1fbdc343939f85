// nls_warp.cuh -- one instance per warp segment of L = 8, 16 or 32 lanes,
// for n <= L (runtime n).
//
// Lane r of a segment owns component r of u and F (FP64) and row r of the
// Jacobian (FP64, or FP32 with NLS_MIXED) in registers.  Row r of J comes
// from forward-mode duals over the variables F_r depends on (Sec. 2.4: the
// stencil of F_r), scattered into the row; the cubic's linear part gives its
// coefficients directly.  The Newton system is solved with an LU with
// partial pivoting (Sec. 3.2) in which rows never move between lanes: each
// lane keeps the position its row would have after the row interchanges, so
// the pivot at step k is the first position >= k holding the largest
// |a_ik| -- the same choice as with explicit swaps.  The pivot row is
// broadcast through shared memory, the right-hand side is eliminated on the
// fly, and back substitution broadcasts one solution component per step.
//
// What bounds it.  FP64: the FP64 pipe.  A warp's FP64 instruction holds its
// scheduler's unit for 64 cycles (76 for a plain add or multiply) however many
// lanes are active (measured: 1 and 32 active lanes alike), so what counts is
// the number of FP64 instructions: columns at and beyond n are skipped by
// warp-uniform branches, and the stencil families' J^T F and J g take their
// three terms.  Mixed: issue slots and dependent latency, so the pivot row
// moves in 16-byte accesses, the pivot search takes one or two redux.sync and
// the loop over the steps is not unrolled (the row shifts by one column per
// step, which keeps every register index a constant), so it stays in the
// instruction cache.
//
// All segments of a warp execute each pass in lock step (idle segments run
// masked); a persistent launch refills idle segments from a work counter.
// The globalisations are those of the thread tiling: Newton (Eq. 2),
// backtracking on Eq. 8-9, dogleg trust region with Eq. 13-15.
#pragma once

#include "nls_common.cuh"

namespace nls {

// Threads per CTA; its warps never wait on each other.  Two warps, so that a
// batch of about a wave spreads evenly (1,000 FP64 n = 32 systems: 309 us, 350
// with four); four with 16 FP64 lanes, whose instances are short: a flush of many
// small requests launches half the CTAs (8,192 FP64 systems of n = 2..16 by
// Newton 479 -> 446 us, by backtracking 485 -> 447; n = 2..12 382 -> 363).  Not
// Rosenbrock's, whose pass counts spread widely (1,024 of n = 10: 1,323 us, 1,343
// with four).
template <int L, int FAM, bool MIXED>
constexpr int warp_tpb() { return L == 16 && !MIXED && FAM != FAM_ROSENBROCK ? 128 : 64; }

// One segment's shared memory.  U holds the pivot row of every step k, from
// its column k on (the factor U by positions), at slot VEC - 1 + (column - k),
// its right-hand side one slot before: the columns right of the pivot start
// on a 16-byte boundary, and the entries (q, c) of one column c lie US - 1 (an
// odd number) apart, so the back substitution's column read is free of bank
// conflicts.  Its space also serves the transposes (tr).  The cubic's A stays
// here rather than in registers: 64 registers fewer per lane let three warps
// instead of two share a scheduler.
template <int L, bool MIXED, int FAM>
struct alignas(16) WarpSmem {
    using P = typename std::conditional<MIXED, float, double>::type;
    static constexpr int VEC = 16 / (int)sizeof(P);
    static constexpr int US = L + VEC;
    static constexpr int AS = L + 2;
    static constexpr int AR = FAM == FAM_CUBIC ? L : 1;
    double u[L];   // u broadcast (residual)
    P vec[L];      // g broadcast
    P prow[L + VEC]; // pivot row + its right-hand side (two-solve solvers)
    union {
        alignas(16) P U[L][US];
        P tr[L][L + 1]; // J^T F transpose-sum
    };
    alignas(16) double A[AR][AS]; // cubic: row r of A (FP64)
};

// Butterfly reductions inside a segment of L lanes (xor offsets < L never
// leave the segment).  `mask` names the lanes executing the call; it is a
// union of whole segments.  Every lane ends with the same bits.
template <int L, class T>
NLS_DI T seg_sum(T v, unsigned mask)
{
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}
template <int L>
NLS_DI uint64_t seg_max(uint64_t v, unsigned mask)
{
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        const uint64_t w = __shfl_xor_sync(mask, v, o);
        v = w > v ? w : v;
    }
    return v;
}
template <int L>
NLS_DI uint32_t seg_max(uint32_t v, unsigned mask)
{
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(mask, v, o));
    return v;
}
// Largest v of each segment, all 32 lanes taking part: one redux.sync when
// the segment is the warp (as cheap as one shuffle).
template <int L>
NLS_DI uint32_t seg_top(uint32_t v)
{
    if constexpr (L == 32) return __reduce_max_sync(0xffffffffu, v);
    else return seg_max<L>(v, 0xffffffffu);
}
template <int L>
NLS_DI uint64_t seg_top(uint64_t v)
{
    const uint32_t h = seg_top<L>((uint32_t)(v >> 32));
    const uint32_t l = seg_top<L>((uint32_t)(v >> 32) == h ? (uint32_t)v : 0u);
    return ((uint64_t)h << 32) | l;
}

template <int L, int FAM, bool MIXED>
struct WarpSolver {
    using P = typename std::conditional<MIXED, float, double>::type;
    using K = decltype(mag_bits(P(0)));
    using SM = WarpSmem<L, MIXED, FAM>;
    static constexpr int VEC = SM::VEC;
    static constexpr int FAMILY = FAM;

    // ---- per-lane data of the current instance
    int r;         // row owned by this lane (0..L-1)
    int n;         // system size
    int lane0;     // first lane of the segment in the warp
    float arowf[FAM == FAM_CUBIC && MIXED ? L : 1];  // cubic, mixed: FP32 copy of row r of A (Jacobian)
    double b_r;                 // cubic: b_r; square: p_r; Bratu: lambda
    double u, F, dN;
    uint64_t fmag;              // max_r |F_r| as a bit pattern (segment-uniform)
    P g, Jg, Fp;
    double fF, Delta;
    int it, nfev, rej, status;
    int ngrad; // trust region: passes that formed g = J^T F and J g
    bool need_jac;

    NLS_DI bool row_live() const { return r < n; }

    // F_r(u) in FP64; all lanes of the segment call it together
    NLS_DI double residual(const double ur, SM &sm, unsigned mask) const
    {
        double f = 0.0;
        if constexpr (FAM == FAM_CUBIC) {
            sm.u[r] = ur;
            __syncwarp(mask);
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < L; j += 2) {
                if (j >= n) break;
                const double2 a = *reinterpret_cast<const double2 *>(&sm.A[r][j]);
                const double2 v = *reinterpret_cast<const double2 *>(&sm.u[j]);
                s = fma(a.x, v.x, s);
                if (j + 1 < n) s = fma(a.y, v.y, s);
            }
            __syncwarp(mask);
            f = s + ur * ur * ur - b_r;
        } else if constexpr (FAM == FAM_BRATU) {
            const double inv_h2 = double((n + 1) * (n + 1));
            double left = __shfl_up_sync(mask, ur, 1, L);
            double right = __shfl_down_sync(mask, ur, 1, L);
            if (r == 0) left = 0.0;
            if (r >= n - 1) right = 0.0;
            f = inv_h2 * ((left + (-2.0) * ur) + right) + b_r * exp(ur);
        } else if constexpr (FAM == FAM_SQUARE) {
            f = ur * ur - b_r;
        } else {
            const double left = __shfl_up_sync(mask, ur, 1, L);
            f = (r == 0) ? 1.0 - ur : 10.0 * (ur - left * left);
        }
        return row_live() ? f : 0.0;
    }

    // partials of F_r over its stencil by forward-mode duals: d0 = dF_r/du_{r-1},
    // d1 = dF_r/du_r, d2 = dF_r/du_{r+1}; 0 where the variable does not exist.
    // Cubic: d1 is the nonlinear part's 3 u_r^2 alone.  All 32 lanes call it.
    NLS_DI void stencil(P &d0, P &d1, P &d2) const
    {
        const P ur = P(u);
        d0 = d1 = d2 = P(0);
        if constexpr (FAM == FAM_CUBIC) {
            const auto x = seed<1, 0, P>(ur);
            d1 = (x * x * x).d[0];
        } else if constexpr (FAM == FAM_BRATU) {
            const P inv_h2 = P((n + 1) * (n + 1));
            const P lam = P(b_r);
            // F_r = (u_{r-1} - 2 u_r + u_{r+1}) / h^2 + lambda e^{u_r}; seeds: 0 left, 1 centre, 2 right
            const auto xl = seed<3, 0, P>(P(0));
            const auto xc = seed<3, 1, P>(ur);
            const auto xr = seed<3, 2, P>(P(0));
            const auto f = inv_h2 * ((xl + P(-2) * xc) + xr) + lam * exp(xc);
            d0 = r > 0 ? f.d[0] : P(0);
            d1 = f.d[1];
            d2 = r + 1 < n ? f.d[2] : P(0);
        } else if constexpr (FAM == FAM_SQUARE) {
            const auto x = seed<1, 0, P>(ur);
            d1 = (x * x).d[0];
        } else {
            // F_0 = 1 - u_0; F_r = 10 (u_r - u_{r-1}^2); seeds: 0 left, 1 centre
            const P ul = __shfl_up_sync(0xffffffffu, ur, 1, L);
            const auto xl = seed<2, 0, P>(ul);
            const auto xc = seed<2, 1, P>(ur);
            const auto f = P(10) * (xc - xl * xl);
            d0 = r > 0 ? f.d[0] : P(0);
            d1 = r > 0 ? f.d[1] : P(-1);
        }
        if (!row_live()) d0 = d1 = d2 = P(0);
    }

    // row r of J(u) in precision P from the stencil's partials
    NLS_DI void jacobian_row(P (&a)[L], const SM &sm, P d0, P d1, P d2) const
    {
        if constexpr (FAM == FAM_CUBIC) {
            // linear coefficients of F_r, plus d(u_r^3)/du_r on the diagonal (FP64:
            // added once, not in every column under a select).  Mixed: added to
            // every column (0 off the diagonal) with 32 lanes, which keeps the copy
            // of the row in registers (2^16 n = 32 systems 3.00 -> 2.91 ms); the
            // select, which the compiler answers with a copy in local memory and
            // half the registers, is the better one below (uneven 2^18 mix 2.77 ->
            // 2.71 ms)
            P diag = P(0);
            if constexpr (!MIXED) diag = sm.A[r][r] + d1;
#pragma unroll
            for (int j = 0; j < L; ++j) {
                P v;
                if constexpr (MIXED && L == 32) v = arowf[j] + ((j == r) ? d1 : 0.f);
                else if constexpr (MIXED) v = (j == r) ? arowf[j] + d1 : arowf[j];
                else v = (j == r) ? diag : sm.A[r][j];
                a[j] = (j < n && row_live()) ? v : P(0);
            }
        } else {
#pragma unroll
            for (int j = 0; j < L; ++j) a[j] = j == r ? d1 : j == r - 1 ? d0 : j == r + 1 ? d2 : P(0);
        }
    }
    NLS_DI void jacobian_row(P (&a)[L], const SM &sm) const
    {
        P d0, d1, d2;
        stencil(d0, d1, d2);
        jacobian_row(a, sm, d0, d1, d2);
    }

    // g = J^T F and J g for the row a (and stencil d0, d1, d2) of this lane
    NLS_DI void gradient(const P (&a)[L], P d0, P d1, P d2, P fp, P &gr, P &Jgr, SM &sm) const
    {
        const unsigned FULL = 0xffffffffu;
        if constexpr (FAM == FAM_CUBIC) {
            // column sums of F_i * row i.  FP64 keeps the products unrounded (one
            // fused instruction per row instead of a multiply and an add)
            P s = P(0);
            if constexpr (MIXED) {
#pragma unroll
                for (int j = 0; j < L; ++j)
                    if (j < n) sm.tr[r][j] = a[j] * fp;
                __syncwarp();
                for (int i = 0; i < n; ++i) s += sm.tr[i][r];
            } else {
#pragma unroll
                for (int j = 0; j < L; ++j)
                    if (j < n) sm.tr[r][j] = a[j];
                sm.vec[r] = fp;
                __syncwarp();
                for (int i = 0; i < n; ++i) s = fma(sm.tr[i][r], sm.vec[i], s);
                __syncwarp();
            }
            gr = row_live() ? s : P(0);
            sm.vec[r] = gr;
            __syncwarp();
            P t = P(0);
#pragma unroll
            for (int j = 0; j < L; ++j)
                if (j < n) t = fma(a[j], sm.vec[j], t);
            Jgr = t;
            __syncwarp();
        } else {
            // three terms at most, in the dense sum's order
            const P q0 = d0 * fp, q1 = d1 * fp, q2 = d2 * fp;
            const P up = __shfl_up_sync(FULL, q2, 1, L);
            const P dn = __shfl_down_sync(FULL, q0, 1, L);
            P s = r > 0 ? up : P(0);
            s += q1;
            if (r + 1 < L) s += dn;
            gr = row_live() ? s : P(0);
            const P gl = __shfl_up_sync(FULL, gr, 1, L), gn = __shfl_down_sync(FULL, gr, 1, L);
            P t = r > 0 ? d0 * gl : P(0);
            t = fma(d1, gr, t);
            Jgr = r + 1 < L ? fma(d2, gn, t) : t;
        }
    }

    // The lane of this lane's segment that holds the pivot of step k: the
    // largest |a| among the rows left (those at positions >= k), the lowest
    // position among equals; a NaN not at position k is never chosen.  One
    // holder of the largest high word decides (kh, h: this lane's word and the
    // largest, from pivot_word); equals, infinities and NaN take the full
    // comparison.  All lanes call it.
    NLS_DI int pivot_lane(P a, uint32_t kh, uint32_t h, int k, int pos, bool left) const
    {
        const unsigned FULL = 0xffffffffu;
        const unsigned seg = L == 32 ? FULL : ((1u << (L & 31)) - 1u) << lane0;
        const K inf = inf_bits(P(0));
        K m = mag_bits(a);
        const uint32_t inf_word = sizeof(K) == 8 ? (uint32_t)((uint64_t)inf >> 32) : (uint32_t)inf;
        unsigned b = __ballot_sync(FULL, kh == h) & seg;
        bool more = (b & (b - 1u)) != 0u || h > inf_word;
        if constexpr (L < 32) more = __any_sync(FULL, more);
        if (more) {
            if (pos > k && m > inf) m = K(0);
            const uint32_t gh = left ? (uint32_t)(sizeof(K) == 8 ? (uint64_t)m >> 32 : (uint64_t)m) + 1u : 0u;
            const uint32_t g = seg_top<L>(gh);
            bool top = left && gh == g;
            if constexpr (sizeof(K) == 8) {
                const uint32_t kl = top ? (uint32_t)m : 0u;
                const uint32_t l = seg_top<L>(kl);
                top = top && kl == l;
            }
            const uint32_t kp = top ? ~(uint32_t)pos : 0u;
            const uint32_t q = seg_top<L>(kp);
            b = __ballot_sync(FULL, top && kp == q) & seg;
        }
        return __ffs(b) - 1;
    }

    // The magnitude's high word + 1 of a candidate (0: none) and the segment's largest.
    NLS_DI static void pivot_word(P a, bool left, uint32_t &kh, uint32_t &h)
    {
        const K m = mag_bits(a);
        kh = left ? (uint32_t)(sizeof(K) == 8 ? (uint64_t)m >> 32 : (uint64_t)m) + 1u : 0u;
        h = seg_top<L>(kh); // every lane, candidate or not
    }

    // One step of the LU at column k.  a[0] is column k of the lane's row and
    // a[c] column k + c; m = n - 1 - k columns follow the pivot.  The updated
    // column k + c goes to a[c - S]: S = 1 moves the row one column to the left.
    // Whole chunks of columns are skipped past n: FP32 eight at a time (fewer
    // tests), FP64 one pair.  In FP64 the next step's search (kh, h) starts as soon
    // as its column is updated, so the reduction runs behind the other columns'
    // updates (20,011 n = 27 systems: 5.18 -> 4.92 ms); the mixed loop, bound by
    // its instructions, ran 6% slower that way in a flush of many sizes.
    template <int S, int W, class SMT>
    NLS_DI void lu_step(P *a, P &b, int k, int m, int &pos, bool &left, bool &ok, uint32_t &kh, uint32_t &h,
                        SMT &sm) const
    {
        constexpr int SKIP = VEC == 4 ? 8 : 2;
        const unsigned FULL = 0xffffffffu;
        const K inf = inf_bits(P(0));
        const int lane = lane0 + r;
        if constexpr (VEC == 4) pivot_word(a[0], left, kh, h);
        const int src = pivot_lane(a[0], kh, h, k, pos, left);
        const int ppos = __shfl_sync(FULL, pos, src);
        P *const row = sm.U[k];
        if (lane == src) {
            if constexpr (VEC == 4) *reinterpret_cast<float2 *>(row + 2) = make_float2(b, a[0]);
            else *reinterpret_cast<double2 *>(row) = make_double2(b, a[0]);
#pragma unroll
            for (int c = 1; c < W; c += VEC) {
                if ((c - 1) % SKIP == 0 && c > m) break;
                if constexpr (VEC == 4)
                    *reinterpret_cast<float4 *>(row + 3 + c) =
                        make_float4(a[c], c + 1 < W ? a[c + 1 < W ? c + 1 : 0] : P(0),
                                    c + 2 < W ? a[c + 2 < W ? c + 2 : 0] : P(0), c + 3 < W ? a[c + 3 < W ? c + 3 : 0] : P(0));
                else
                    *reinterpret_cast<double2 *>(row + 1 + c) =
                        make_double2(a[c], c + 1 < W ? a[c + 1 < W ? c + 1 : 0] : P(0));
            }
        }
        __syncwarp();
        P p0, pb;
        if constexpr (VEC == 4) {
            const float2 v = *reinterpret_cast<const float2 *>(row + 2);
            pb = v.x;
            p0 = v.y;
        } else {
            const double2 v = *reinterpret_cast<const double2 *>(row);
            pb = v.x;
            p0 = v.y;
        }
        const K pm = mag_bits(p0);
        if (pm == K(0) || pm >= inf) ok = false;
        const P pr = rcp(p0);
        if (r == 0) sm.vec[k] = pr;
        // the row at position k moves to the pivot's old position
        if (left && pos == k) pos = ppos;
        if (lane == src) {
            pos = k;
            left = false;
        }
        const P l = left ? a[0] * pr : P(0);
#pragma unroll
        for (int c = 1; c < W; c += VEC) {
            if ((c - 1) % SKIP == 0 && c > m) break;
            if constexpr (VEC == 4) {
                const float4 v = *reinterpret_cast<const float4 *>(row + 3 + c);
                a[c - S] = a[c] - l * v.x;
                if (c + 1 < W) a[c + 1 - S] = a[c + 1] - l * v.y;
                if (c + 2 < W) a[c + 2 - S] = a[c + 2] - l * v.z;
                if (c + 3 < W) a[c + 3 - S] = a[c + 3] - l * v.w;
            } else {
                const double2 v = *reinterpret_cast<const double2 *>(row + 1 + c);
                a[c - S] = a[c] - l * v.x;
                if (c == 1) pivot_word(a[1 - S], left, kh, h);
                if (c + 1 < W && c + 1 <= m) a[c + 1 - S] = a[c + 1] - l * v.y;
            }
        }
        b -= l * pb;
    }

    // LU with partial pivoting and on-the-fly elimination of b; on return
    // b holds x_r (component r of the solution) in lane r.  Returns false
    // (segment-uniform) on a zero or non-finite pivot.  The row a is consumed.
    // FP32: the steps are a loop whose body moves the row one column to the
    // left, so it fits the instruction cache.  FP64: the steps are unrolled and
    // the row stays in place; a shifting update would overwrite a register that
    // the FP64 unit, which reads its operands late, still has to fetch (the
    // shifting loop measured 6.98 ms on 20,011 trust-region n = 27 systems).
    // Against whole rows written by scalar stores, 64-bit shuffle butterflies
    // for the pivot and unskipped columns: 2^16 mixed n = 32 systems
    // (backtracking) 5.66 -> 2.92 ms, 20,011 FP64 n = 27 ones (trust region) 6.61
    // -> 4.92 ms, 1,024 ten-dimensional Rosenbrock ones 2.72 -> 1.83 ms.
    template <class SMT>
    NLS_DI bool lu_solve(P (&a)[L], P &b, SMT &sm) const
    {
        const unsigned FULL = 0xffffffffu;
        int pos = r;              // position of this lane's row after the interchanges
        bool left = row_live();   // not a pivot row yet
        bool ok = true;
        uint32_t kh = 0, h = 0;
        if constexpr (!MIXED) pivot_word(a[0], left, kh, h);
        if constexpr (MIXED) {
            for (int k = 0; k < n; ++k) lu_step<1, L>(a, b, k, n - 1 - k, pos, left, ok, kh, h, sm);
        } else {
            static_for<0, L>([&](auto Kc) {
                constexpr int k = decltype(Kc)::value;
                if (k < n) lu_step<0, L - k>(a + k, b, k, n - 1 - k, pos, left, ok, kh, h, sm);
            });
        }
        __syncwarp(); // the reciprocals are written
        // back substitution: lane k takes pivot row k's right-hand side and
        // reciprocal; x_k goes to every lane, and the lanes of earlier positions
        // remove its contribution
        const bool live = row_live();
        P y = live ? sm.U[r][VEC - 2] : P(0);
        const P rk = live ? sm.vec[r] : P(0);
#pragma unroll 4
        for (int k = n - 1; k > 0; --k) {
            const P xk = __shfl_sync(FULL, y * rk, k, L);
            if (r < k) y -= sm.U[r][VEC - 1 + k - r] * xk;
        }
        __syncwarp(); // U is free for the next use
        b = y * rk;
        return ok;
    }

    // Load instance k and test u0; executed by the lanes in `mask` (whole segments).
    NLS_DI void init(const SolveArgs &a, int64_t k, SM &sm, unsigned mask)
    {
        const int64_t B = a.ld;
        b_r = 0.0;
        if constexpr (FAM == FAM_CUBIC) {
#pragma unroll
            for (int j = 0; j < L; ++j) {
                double v = 0.0;
                if (j < n && row_live()) v = __ldg(a.params + (int64_t)(r * n + j) * B + k);
                sm.A[r][j] = v;
                if constexpr (MIXED) arowf[j] = float(v);
            }
            if (row_live()) b_r = __ldg(a.params + (int64_t)(n * n + r) * B + k);
        } else if constexpr (FAM == FAM_BRATU) {
            b_r = __ldg(a.params + k);
        } else if constexpr (FAM == FAM_SQUARE) {
            if (row_live()) b_r = __ldg(a.params + (int64_t)r * B + k);
        }
        u = row_live() ? a.u[(int64_t)r * B + k] : 0.0;
        F = residual(u, sm, mask);
        dN = 0.0;
        nfev = 1;
        it = 0;
        rej = 0;
        ngrad = 0;
        Delta = TR_DELTA0;
        need_jac = true;
        fF = seg_sum<L>(F * F, mask);
        fmag = seg_max<L>(mag_bits(F), mask);
        if (fmag >= INF64_BITS) status = ST_NONFINITE;
        else if (fmag <= mag_bits(a.abstol)) status = ST_SUCCESS;
        else if (a.maxiters <= 0) status = ST_MAXITERS;
        else status = ST_RUNNING;
    }

    // Write instance k's results (no cross-lane communication).
    NLS_DI void finish(const SolveArgs &a, int64_t k) const
    {
        if (row_live()) a.u[(int64_t)r * a.ld + k] = u;
        if (r == 0) {
            if (a.status) a.status[k] = status;
            if (a.iters) a.iters[k] = it;
            if (a.resid) a.resid[k] = bits_to_double(fmag);
            if (a.nfev) a.nfev[k] = nfev;
            if (a.ngrad) a.ngrad[k] = ngrad;
        }
    }

    // One pass; `run` is false for idle segments, which execute the same
    // instructions (lock step) without changing their state.
    NLS_DI void pass(const SolveArgs &A, SM &sm, bool run)
    {
        if (run) ++it;
        bool failed = false;
        if (__any_sync(0xffffffffu, run && need_jac)) {
            const bool fresh = run && need_jac;
            P a[L], d0, d1, d2;
            stencil(d0, d1, d2);
            jacobian_row(a, sm, d0, d1, d2);
            const P fp = P(F);
            if (fresh) Fp = fp;
            if (A.alg == ALG_TRUST_DOGLEG) {
                P gr, Jgr;
                gradient(a, d0, d1, d2, fp, gr, Jgr, sm);
                if (fresh) {
                    g = gr;
                    Jg = Jgr;
                    ++ngrad;
                }
            }
            P b = -fp;
            const bool ok = lu_solve(a, b, sm);
            if (fresh) {
                if (!ok) {
                    status = ST_SINGULAR;
                    failed = true;
                } else {
                    dN = row_live() ? double(b) : 0.0;
                    need_jac = false;
                }
            }
        }
        const bool go = run && !failed;

        if (A.alg == ALG_NEWTON) {
            const double un = u + dN;
            const double Fn = residual(un, sm, 0xffffffffu);
            if (go) {
                u = un;
                F = Fn;
                ++nfev;
                need_jac = true;
            }
        } else if (A.alg == ALG_NEWTON_BACKTRACK) {
            // slope F^T J dN of Eq. 9 by linearity: J dN = -F, so it is -||F||^2
            const double s = -fF;
            const double phi0 = 0.5 * fF;
            double alpha = 1.0;
            bool trying = go, ok = false;
            for (int m = 0; m < LS_MAX_TRIALS; ++m) {
                if (!__any_sync(0xffffffffu, trying)) break;
                const double ut = fma(alpha, dN, u);
                const double Ft = residual(ut, sm, 0xffffffffu);
                const double fFt = seg_sum<L>(Ft * Ft, 0xffffffffu);
                const bool fin = seg_all(mag_bits(Ft) < INF64_BITS);
                if (trying) {
                    ++nfev;
                    if (fin && 0.5 * fFt <= phi0 + LS_C1 * alpha * s) {
                        u = ut;
                        F = Ft;
                        fF = fFt;
                        ok = true;
                        trying = false;
                    }
                }
                alpha *= LS_RHO;
            }
            if (go) {
                if (!ok) {
                    status = ST_LS_FAILED;
                    failed = true;
                } else {
                    need_jac = true;
                }
            }
        } else {
            // Every reduction is taken by all segments of the warp before any
            // per-segment branch (segments of one warp may take different
            // dogleg branches; a collective inside a branch would diverge).
            const P D2 = P(Delta * Delta);
            const P nN2 = seg_sum<L>(P(dN) * P(dN), 0xffffffffu);
            // pred = -2 F.Jd - ||Jd||^2 (Eq. 15) from segment-uniform scalars:
            // J dN = -F and F.(J g) = g.g (g = J^T F), so no J d is formed
            double d = dN, pred = fF;
            // the dogleg's sums and quotients only when a segment's Newton step
            // leaves its region (a warp-uniform branch)
            if (__any_sync(0xffffffffu, run && !(nN2 <= D2))) {
                const P gg = seg_sum<L>(g * g, 0xffffffffu);
                const P JgJg = seg_sum<L>(Jg * Jg, 0xffffffffu);
                const P t = gg / JgJg; // Cauchy point c = -t g minimises the model along -g
                const P cc = t * t * gg;
                const P w = P(dN) + t * g; // dN - c
                const P aa = seg_sum<L>(w * w, 0xffffffffu);
                const P bb = seg_sum<L>(-t * g * w, 0xffffffffu);
                if (nN2 <= D2) {
                    // the Newton step
                } else if (cc >= D2) {
                    const P sc = P(Delta) / nls_sqrt(gg);
                    d = double(-sc * g);
                    pred = double(sc * (P(2) * gg - sc * JgJg));
                } else {
                    const P q = cc - D2;
                    const P tau = (-bb + nls_sqrt(bb * bb - aa * q)) / aa;
                    d = double(fma(tau, w, -t * g));
                    const P s1 = (P(1) - tau) * t; // J d = -s1 J g - tau F
                    pred = double(s1 * (P(2) * (P(1) - tau) * gg - s1 * JgJg) + tau * (P(2) - tau) * P(fF));
                }
            }
            if (!row_live()) d = 0.0;
            const double ut = u + d;
            const double Ft = residual(ut, sm, 0xffffffffu);
            const double fFt = seg_sum<L>(Ft * Ft, 0xffffffffu);
            const bool fin = seg_all(mag_bits(Ft) < INF64_BITS);
            const double ared = fF - fFt;
            if (go) {
                ++nfev;
                if (tr_step_outcome(A.tr_scheme, pred > 0.0 && fin, ared, pred, !(nN2 <= D2), Delta)) {
                    u = ut;
                    F = Ft;
                    fF = fFt;
                    need_jac = true;
                    rej = 0;
                } else {
                    if (++rej >= TR_MAX_REJECTIONS) {
                        status = ST_TR_STALLED;
                        failed = true;
                    }
                }
            }
        }
        const bool fin = seg_all(mag_bits(F) < INF64_BITS);
        const bool conv = seg_all(mag_bits(F) <= mag_bits(A.abstol));
        if (go && !failed) {
            if (!fin) status = ST_NONFINITE;
            else if (conv) status = ST_SUCCESS;
            else if (it >= A.maxiters) status = ST_MAXITERS;
        }
        // the residual's norm itself is an output: formed when an instance ends
        if (__any_sync(0xffffffffu, run && status != ST_RUNNING)) residual_norm(run);
    }

    // whether p holds on every lane of this lane's segment (all lanes call it)
    NLS_DI bool seg_all(bool p) const
    {
        const unsigned b = __ballot_sync(0xffffffffu, p);
        return L == 32 ? b == 0xffffffffu : ((b >> lane0) & ((1u << (L & 31)) - 1u)) == (1u << (L & 31)) - 1u;
    }
    // fmag = max_r |F_r| for the segments with `run` (all lanes call it)
    NLS_DI void residual_norm(bool run)
    {
        const uint64_t m = seg_top<L>(mag_bits(F));
        if (run) fmag = m;
    }
};

template <int L, bool MIXED, int FAM>
constexpr int warp_smem_bytes()
{
    constexpr int bytes = (warp_tpb<L, FAM, MIXED>() / 32) * (32 / L) * (int)sizeof(WarpSmem<L, MIXED, FAM>);
    static_assert(bytes <= 48 * 1024, "no opt-in beyond 48 KB is made for these kernels");
    return bytes;
}

// The segment loop shared by the warp-tiled solvers S (r, n, lane0, status,
// init / pass / finish): segments take instances from the work counter (or
// the static slot), every pass runs in lock step over the whole warp.
template <class S, int L, bool MIXED>
NLS_DI void warp_lanes(SolveArgs &a)
{
    apply_dyn_batch(a);
    using SM = typename S::SM;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int SEGS = 32 / L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int seg = lane / L;
    SM &sm = reinterpret_cast<SM *>(smem_raw)[warp * SEGS + seg];
    const unsigned FULL = 0xffffffffu;

    const unsigned long long t_end = a.budget_ns ? global_ns() + a.budget_ns : ~0ull;
    S s;
    s.r = lane % L;
    s.n = a.n;
    s.lane0 = seg * L;
    s.status = ST_ABORTED;
    bool have = false, exhausted = false, first = true;
    int64_t k = -1;
    unsigned long long local_solved = 0;
    const int64_t warp_global = (int64_t)blockIdx.x * (warp_tpb<L, S::FAMILY, MIXED>() / 32) + warp;

    for (;;) {
        // segments are the units of work: one ballot bit per segment leader
        const unsigned seg_live = __ballot_sync(FULL, have && s.r == 0);
        const int live = __popc(seg_live);
        if (!exhausted && live <= (SEGS > 1 ? SEGS - 1 : 0)) {
            const bool want = !have;
            int64_t cand = a.batch;
            if (a.counter == nullptr) {
                if (first && want) cand = warp_global * SEGS + seg;
            } else {
                const unsigned m = __ballot_sync(FULL, want && s.r == 0);
                const int leader = m ? __ffs(m) - 1 : 0;
                unsigned long long base = 0;
                if (lane == leader && m) base = atomicAdd(a.counter, (unsigned long long)__popc(m));
                base = __shfl_sync(FULL, base, leader);
                if (want) cand = (int64_t)base + __popc(m & ((1u << (seg * L)) - 1u));
            }
            first = false;
            const bool got = want && cand < a.batch;
            // the lanes of segments that got an instance load it together
            const unsigned gm = __ballot_sync(FULL, got);
            if (got) {
                k = cand;
                s.init(a, k, sm, gm);
                if (s.status != ST_RUNNING) {
                    s.finish(a, k);
                    local_solved += (s.status == ST_SUCCESS && s.r == 0);
                } else {
                    have = true;
                }
            }
            exhausted = (a.counter == nullptr) || __any_sync(FULL, want && !got);
        }
        if (!__any_sync(FULL, have)) {
            if (exhausted) break;
            continue;
        }
        // the deadline test is warp-uniform (lane 0's clock), so skipping the
        // pass never splits a collective
        const bool late = a.budget_ns && __shfl_sync(FULL, global_ns(), 0) > t_end;
        if (late) {
            s.residual_norm(have);
            if (have) s.status = ST_ABORTED;
        } else {
            s.pass(a, sm, have);
        }
        if (have && s.status != ST_RUNNING) {
            s.finish(a, k);
            local_solved += (s.status == ST_SUCCESS && s.r == 0);
            have = false;
        }
    }
    if (a.solved) {
        unsigned long long t = local_solved;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
        if (lane == 0 && t) atomicAdd(a.solved, t);
    }
}

// CTAs per SM that the compiler makes room for (0: its own choice).  The
// 32-lane FP64 kernels take the 6 that the cubic's shared memory allows (164
// registers instead of 222, which held 4: 5,000 n = 27 systems 916 us against
// 1,151).  Mixed, 8 CTAs (128 registers and a spill) measured 2% faster on n = 32
// alone but 5% slower in a flush of many sizes.  16 lanes: sixteen FP64 warps per
// SM (120 registers; left alone, Bratu's kernel took 154, which held twelve), and
// 24 mixed ones of the families without a matrix of their own (80 registers
// instead of 89 to 96; 20,000 systems of n = 16: square 196 -> 184 us, Bratu 175 ->
// 171).
template <int L, int FAM, bool MIXED>
constexpr int warp_min_ctas()
{
    if (L == 32) return MIXED ? 0 : 6;
    if (L == 16 && MIXED) return FAM == FAM_CUBIC ? 0 : 12;
    if (L == 16) return FAM == FAM_ROSENBROCK ? 0 : 4;
    return 0;
}

template <int L, int FAM, bool MIXED>
__global__ void __launch_bounds__((warp_tpb<L, FAM, MIXED>()), (warp_min_ctas<L, FAM, MIXED>())) k_solve_warp(SolveArgs a)
{
    warp_lanes<WarpSolver<L, FAM, MIXED>, L, MIXED>(a);
}

} // namespace nls
