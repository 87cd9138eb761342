// lp_fp64_simplex.cu -- FP64 dense simplex, one CTA per LP: small tableaux are
// resident in shared memory (fp64_resident_kernel, solve_one below); larger
// ones are never updated as a whole (fp64_deferred_kernel, persistent CTAs
// taking LPs from an atomic counter; lp_fp64_deferred.cuh).
//
// Method: Gurung & Ray, "Simultaneous Solving of Batched Linear Programs on a
// GPU" (arXiv 1802.08557).  Section 4.1 assigns one CUDA block per LP; Section
// 4.2 parallelises Step 1 (entering variable) and Step 2 (leaving variable) as
// reductions and Step 3 (pivot) over the tableau elements.  Differences from
// the paper's kernel (which kept the full tableau in global memory and used
// shared/global tree reductions):
//  - the condensed (Tucker) tableau is kept: one column per NON-basic
//    variable plus the right-hand side (column 0).  A pivot swaps the labels of
//    the entering column and the leaving row.  Basic columns of the paper's
//    full tableau are unit vectors and carry no information;
//  - the tableau lives in shared memory for the whole solve (global memory is
//    touched only to read A, b, c and write the results); above a size,
//    elements are formed only when a pivot reads them (deferred updates);
//  - reductions are warp `redux` instructions on 64-bit order-preserving
//    integer keys of the FP64 values (exact, no FP64-pipe compares);
//  - phase I runs in the same kernel (the paper launches twice, Section 5);
//  - Steps 1 and 2 screen their candidates without FP64 arithmetic (the FP64
//    pipe of GB300 is ~60x slower than FP32 and a warp FP64 instruction costs
//    the whole warp's pipe time whatever its active mask): Step 1 bounds the tie
//    window of the minimum reduced cost in units of the integer key, Step 2
//    bounds the ratios in FP32 with a window wider than every FP32 rounding
//    error.  When the screen leaves exactly one candidate it is the exact
//    answer; otherwise the exact FP64 rule runs on the candidates.  The result
//    is the same as the plain rule's in every case.
//
// Arithmetic is the oracle's, operation for operation, so that both reach the
// same pivot sequence: ratio = rhs / t (IEEE divide), pivot row = row / PE
// (IEEE divide), update t_ij = fma(-t_ie, r_j, t_ij), tie window
// v + tau*max(1,|v|) as a product followed by a sum.  This file is compiled
// with --fmad=false and only uses the _rn intrinsics for FP64 arithmetic.

#include <climits>

#include "lp_device.cuh"
#include "lp_fp64_deferred.cuh"
#include "lp_internal.h"

namespace lpb {
namespace {

struct Tab {
    double* T;        // R x LD, row-major; column 0 = right-hand side
    double* colE;     // copy of the pivot column
    int* col_var;     // variable of each column (1..Cvar live)
    int* row_var;     // basic variable of each constraint row
    int LD;
};

// Step 3 (Section 3.1, Listing 1) on the condensed tableau: divide pivot row
// l by PE = colE[l], then t_ij <- fma(-t_ie, r_j, t_ij) for every other active
// row.  In column e (which now holds the leaving variable) the old entry of the
// paper's full tableau is the unit column of a basic variable, i.e. 0 off the
// pivot row and 1 on it, so r_e = 1/PE and t_ie <- fma(-t_ie, r_e, 0).
// colE[0..Ract) must hold column e on entry.  Returns the variable that left
// the basis (now the label of column e), read by every thread between the two
// barriers, where nothing writes it.
// The barrier of the thread group that owns the LP: the CTA, or (kWarp: a
// one-warp CTA) the warp -- no block barrier, shared-memory writes ordered by
// __syncwarp.
template <bool kWarp>
__device__ __forceinline__ void group_sync() {
    if (kWarp) __syncwarp();
    else __syncthreads();
}

template <bool kWarp>
__device__ __forceinline__ int pivot(Tab& tb, int Ract, int Cact, int l, int e) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int LD = tb.LD;
    double* T = tb.T;
    const double* colE = tb.colE;
    const double pe = colE[l];
    double* Tl = T + (size_t)l * LD;
    for (int j = tid; j < Cact; j += nt) {
        const double v = (j == e) ? 1.0 : Tl[j];
        Tl[j] = __ddiv_rn(v, pe);
    }
    if (tid == 0) {
        const int ev = tb.col_var[e];
        tb.col_var[e] = tb.row_var[l];
        tb.row_var[l] = ev;
    }
    group_sync<kWarp>();
    const int left = tb.col_var[e];
    const int total = (Ract - 1) * Cact;
    int ii = tid / Cact;
    int jj = tid - ii * Cact;
    const int di = nt / Cact;
    const int dj = nt - di * Cact;
    for (int idx = tid; idx < total; idx += nt) {
        const int r = ii + (ii >= l ? 1 : 0);
        double* t = T + (size_t)r * LD + jj;
        const double old = (jj == e) ? 0.0 : *t;
        *t = __fma_rn(-colE[r], Tl[jj], old);
        ii += di;
        jj += dj;
        if (jj >= Cact) { jj -= Cact; ++ii; }
    }
    group_sync<kWarp>();
    return left;
}

// A retired artificial (it just left the basis and may never re-enter) sits
// in column e: move the last live column into its place and shrink.
template <bool kWarp>
__device__ __forceinline__ void retire_column(Tab& tb, int Ract, int e, int& Cvar) {
    const int tid = threadIdx.x, nt = blockDim.x;
    if (e != Cvar) {
        for (int r = tid; r < Ract; r += nt) {
            double* row = tb.T + (size_t)r * tb.LD;
            row[e] = row[Cvar];
        }
        if (tid == 0) tb.col_var[e] = tb.col_var[Cvar];
    }
    --Cvar;
    group_sync<kWarp>();
}

// One LP, Steps 1-3 until it halts, in shared memory: the reductions' scratch
// in `small` (SmallLayout), the tableau and its vectors in `big` (big_layout).
template <bool kWarp = false>
__device__ __forceinline__ void solve_one(const DeviceBatch& B, const Tolerances& tol, const int lp,
                                          unsigned char* small, unsigned char* big, int32_t* diag)
{
    const int m = B.m[lp];
    const int n = B.n[lp];
    const int nm = n + m;
    const double* __restrict__ A = B.A + B.a_off[lp];
    const double* __restrict__ bv = B.b + B.b_off[lp];
    const double* __restrict__ cv = B.c + B.c_off[lp];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;

    // k-independent part of the layout (k = 0 gives the same offsets)
    const BigLayout L0 = big_layout(m, n, 0);
    // the group's reductions: block-wide through the scratch in `small`, or
    // (kWarp) `redux` within the one warp
    auto make_red = [&]() {
        if constexpr (kWarp) {
            return WarpGroup();
        } else {
            return Reducer{reinterpret_cast<long long*>(small + SmallLayout::red64),
                           reinterpret_cast<unsigned*>(small + SmallLayout::red32), nw, warp, lane};
        }
    };
    auto red = make_red();
    long long* rkey = reinterpret_cast<long long*>(big + L0.rkey);
    int* row_var = reinterpret_cast<int*>(big + L0.row_var);
    int* neg = reinterpret_cast<int*>(big + L0.neg);

    // ---- Tableau build (the host-side fill of Section 4.1, done here) -----
    // Rows with b_i < 0 are negated and get an artificial (two-phase method,
    // Section 3); they are ranked in ascending row order.
    int k = 0;
    for (int i0 = 0; i0 < m; i0 += nt) {
        const int i = i0 + tid;
        const bool isneg = (i < m) && (bv[i] < 0.0);
        int tot;
        const int r = k + red.prefix_count(isneg, tot);
        if (i < m) {
            if (isneg) {
                neg[r] = i;
                row_var[i] = nm + r;
            } else {
                row_var[i] = n + i;
            }
        }
        k += tot;
    }
    group_sync<kWarp>();  // neg[] and row_var[] are read by other threads below

    const BigLayout L = big_layout(m, n, k);
    Tab tb;
    tb.T = reinterpret_cast<double*>(big + L.T);
    tb.colE = reinterpret_cast<double*>(big + L.colE);
    tb.col_var = reinterpret_cast<int*>(big + L.col_var);
    tb.row_var = row_var;
    tb.LD = L.LD;
    const int LD = L.LD;
    double* T = tb.T;  // the tableau is written through several pointers: no restrict
    int Cvar = n + k;  // live variable columns 1..Cvar

    for (int j = tid; j <= Cvar; j += nt)
        tb.col_var[j] = (j == 0) ? -1 : (j <= n ? j - 1 : n + neg[j - 1 - n]);
    {
        // A into rows 0..m-1, columns 1..n: asynchronous copies, all in flight
        // at once, then the negated rows in place; then b and the slack columns
        const int64_t cnt = (int64_t)m * n;
        int i = tid / n, j = tid - i * n;
        const int di = nt / n, dj = nt - di * n;
        for (int64_t idx = tid; idx < cnt; idx += nt) {
            cp_async8(T + (size_t)i * LD + 1 + j, A + idx);
            i += di;
            j += dj;
            if (j >= n) { j -= n; ++i; }
        }
        cp_async_wait_all();
        group_sync<kWarp>();
        if (k > 0)
            for (int64_t idx = tid; idx < cnt; idx += nt) {
                const int i2 = (int)(idx / n), j2 = (int)(idx - (int64_t)i2 * n);
                if (row_var[i2] >= nm) T[(size_t)i2 * LD + 1 + j2] = -T[(size_t)i2 * LD + 1 + j2];
            }
        for (int r = warp; r < m; r += nw) {
            const bool isneg = row_var[r] >= nm;
            double* Tr = T + (size_t)r * LD;
            for (int t = lane; t <= k; t += 32) {
                const int jj = (t == 0) ? 0 : n + t;
                const double v = (t == 0) ? bv[r] : ((neg[t - 1] == r) ? 1.0 : 0.0);
                Tr[jj] = isneg ? -v : v;
            }
        }
    }
    {
        double* Tm = T + (size_t)m * LD;
        for (int j = tid; j <= Cvar; j += nt) Tm[j] = (j >= 1 && j <= n) ? -cv[j - 1] : 0.0;
    }
    long long bmax_key = 0x3FF0000000000000LL;  // 1.0
    for (int i = tid; i < m; i += nt) bmax_key = max(bmax_key, abskey(bv[i]));
    bmax_key = -red.min_i64(-bmax_key);  // also orders the fills above
    if (k > 0) {
        // auxiliary objective: maximise -(sum of artificials), priced out by
        // subtracting every negated row in ascending row order
        double* Tw = T + (size_t)(m + 1) * LD;
        for (int j = tid; j <= Cvar; j += nt) {
            double w = 0.0;
            for (int t = 0; t < k; ++t) w = __dsub_rn(w, T[(size_t)neg[t] * LD + j]);
            Tw[j] = w;
        }
        group_sync<kWarp>();
    }

    const long long key_neg_eps_opt = okey(-tol.eps_opt);
    const long long key_eps_piv = okey(tol.eps_piv);
    const int max_iters = tol.max_iters > 0 ? tol.max_iters : 50 * (m + n);
    int iters = 0;
    int status = -1;
    int phase = (k > 0) ? 1 : 2;
    int yrow = m;

    while (status < 0) {
        const int orow = (phase == 1) ? m + 1 : m;
        const int Ract = (phase == 1) ? m + 2 : m + 1;
        const double* Trow = T + (size_t)orow * LD;

        // ---- Step 1: entering variable (most negative reduced cost) -------
        long long dloc = LLONG_MAX;
        for (int j = 1 + tid; j <= Cvar; j += nt)
            if (tb.col_var[j] < nm) dloc = min(dloc, okey(Trow[j]));
        const long long dmin = red.min_i64(dloc);
        if (dmin >= key_neg_eps_opt) {
            if (phase == 2) { status = kOptimal; break; }
            // ---- end of phase I (Section 3, two-phase method) -------------
            const double wstar = -T[(size_t)(m + 1) * LD];
            if (wstar > __dmul_rn(tol.eps_feas, __longlong_as_double(bmax_key))) {
                status = kInfeasible;
                yrow = m + 1;
                break;
            }
            // drive artificials still basic (at level 0) out of the basis on
            // the lowest non-artificial column with |t_ij| > eps_piv
            for (int i = 0; i < m && status < 0; ++i) {
                if (row_var[i] < nm) continue;
                const double* Ti = T + (size_t)i * LD;
                unsigned sel = 0xffffffffu;
                for (int j = 1 + tid; j <= Cvar; j += nt)
                    if (tb.col_var[j] < nm && abskey(Ti[j]) > key_eps_piv)
                        sel = min(sel, ((unsigned)tb.col_var[j] << 16) | (unsigned)j);
                sel = red.min_u32(sel);
                if (sel == 0xffffffffu) continue;  // redundant row
                if (iters >= max_iters) { status = kIterLimit; break; }
                const int e = (int)(sel & 0xffffu);
                for (int r = tid; r < m + 1; r += nt) tb.colE[r] = T[(size_t)r * LD + e];
                group_sync<kWarp>();
                const int left = pivot<kWarp>(tb, m + 1, Cvar + 1, i, e);
                ++iters;
                if (left >= nm) retire_column<kWarp>(tb, m + 1, e, Cvar);
            }
            phase = 2;
            continue;
        }
        // screen: columns whose key lies within the tie-window bound of dmin
        const unsigned long long win = step1_window(dmin, tol.key_window);
        unsigned ecnt = 0, esel = 0xffffffffu;
        for (int j = 1 + tid; j <= Cvar; j += nt) {
            const int v = tb.col_var[j];
            if (v < nm && (unsigned long long)okey(Trow[j]) - (unsigned long long)dmin <= win) {
                ++ecnt;
                esel = min(esel, ((unsigned)v << 16) | (unsigned)j);
            }
        }
        red.count_min(ecnt, esel, ecnt, esel);
        if (ecnt > 1) {
            // several candidates: the exact rule (lowest label within the window)
            const long long kthr = okey(tie_threshold(kval(dmin), tol.tau));
            unsigned sel = 0xffffffffu;
            for (int j = 1 + tid; j <= Cvar; j += nt) {
                const int v = tb.col_var[j];
                if (v < nm && okey(Trow[j]) <= kthr) sel = min(sel, ((unsigned)v << 16) | (unsigned)j);
            }
            esel = red.min_u32(sel);
        }
        const int e = (int)(esel & 0xffffu);

        // ---- Step 2: leaving row (minimum ratio rhs_i / t_ie, t_ie > eps) --
        // FP32 screen: rows with both operands in [2^-100, 2^100] (or rhs 0)
        // get a float ratio; the others are always candidates.  The operands
        // are truncated to FP32 by integer operations (< 2^-23 relative
        // each): a hardware conversion would take the FP64 pipe, which bounds
        // this kernel.  The window (far wider than the screen's error) is
        // set below.
        int floc = INT_MAX;
        for (int i = tid; i < Ract; i += nt) {
            const double t = T[(size_t)i * LD + e];
            tb.colE[i] = t;
            if (i < m) {
                long long code = LLONG_MAX;  // not eligible
                if (okey(t) > key_eps_piv) {
                    const double beta = T[(size_t)i * LD];
                    const int et = dexp(t), eb = dexp(beta);
                    const bool safe = et >= -100 && et <= 100 && (abskey(beta) == 0 || (eb >= -100 && eb <= 100));
                    if (safe) {
                        const int fk = fkey(__fdividef(f64_to_f32_trunc(beta), f64_to_f32_trunc(t)));
                        code = fk;
                        floc = min(floc, fk);
                    } else {
                        code = LLONG_MIN;  // unscreened: always a candidate
                    }
                }
                rkey[i] = code;
            }
        }
        const int fmin = red.min_i32(floc);
        long long fwin = LLONG_MIN;
        if (fmin != INT_MAX) {
            const float fm = fval(fmin);
            fwin = fkey(fm + __fmaf_rn(tol.ratio_rel, fabsf(fm), tol.ratio_abs));
        }
        unsigned lcnt = 0, lsel = 0xffffffffu;
        for (int i = tid; i < m; i += nt) {
            const long long code = rkey[i];
            if (code == LLONG_MIN || (code != LLONG_MAX && code <= fwin)) {
                ++lcnt;
                lsel = min(lsel, (unsigned)i);
            }
        }
        red.count_min(lcnt, lsel, lcnt, lsel);
        if (lcnt == 0) {
            status = (phase == 2) ? kUnbounded : kNumerical;
            break;
        }
        if (lcnt > 1) {
            // several candidates: exact ratios of the candidates, exact rule
            long long rloc = LLONG_MAX;
            for (int i = tid; i < m; i += nt) {
                const long long code = rkey[i];
                long long rk = LLONG_MAX;
                if (code == LLONG_MIN || (code != LLONG_MAX && code <= fwin))
                    rk = okey(__ddiv_rn(T[(size_t)i * LD], tb.colE[i]));
                rkey[i] = rk;
                rloc = min(rloc, rk);
            }
            const long long rmin = red.min_i64(rloc);
            const long long rthr = okey(tie_threshold(kval(rmin), tol.tau));
            unsigned sel = 0xffffffffu;
            for (int i = tid; i < m; i += nt)
                if (rkey[i] <= rthr) sel = min(sel, (unsigned)i);
            lsel = red.min_u32(sel);
        }
        const int l = (int)lsel;
        if (abskey(tb.colE[l]) >= 0x7FF0000000000000LL) { status = kNumerical; break; }
        if (iters >= max_iters) { status = kIterLimit; break; }

        // ---- Step 3: pivot ---------------------------------------------------
        const int left = pivot<kWarp>(tb, Ract, Cvar + 1, l, e);
        ++iters;
        if (left >= nm) retire_column<kWarp>(tb, Ract, e, Cvar);
    }

    // ---- labels must name variables (self-check before they index global
    // memory); a failure is recorded and the LP reported as LP_NUMERICAL ----
    {
        unsigned badl = 0, dummy;
        const unsigned nvar = (unsigned)(nm + k);
        for (int i = tid; i < m; i += nt) badl += ((unsigned)row_var[i] >= nvar) ? 1u : 0u;
        for (int j = 1 + tid; j <= Cvar; j += nt) badl += ((unsigned)tb.col_var[j] >= nvar) ? 1u : 0u;
        red.count_min(badl, 0u, badl, dummy);
        if (badl) {
            if (tid == 0) {
                record_internal_error(diag, 6, lp, (int)badl, status, iters, phase, Cvar);
                B.status[lp] = kNumerical;
                B.iters[lp] = iters;
            }
            return;
        }
    }

    // ---- results: x (basic rows -> rhs, non-basic -> 0), y (slack reduced
    // costs of row `yrow`), objective corner, status, pivots -----------------
    double* __restrict__ x = B.x + B.x_off[lp];
    double* __restrict__ y = B.y ? B.y + B.y_off[lp] : nullptr;
    const double* Ty = T + (size_t)yrow * LD;
    for (int j = 1 + tid; j <= Cvar; j += nt) {
        const int v = tb.col_var[j];
        if ((unsigned)v < (unsigned)n) x[v] = 0.0;
        else if (v >= n && v < nm && y) y[v - n] = Ty[j];
    }
    for (int i = tid; i < m; i += nt) {
        const int v = row_var[i];
        if ((unsigned)v < (unsigned)n) x[v] = T[(size_t)i * LD];
        else if (v >= n && v < nm && y) y[v - n] = 0.0;
    }
    if (tid == 0) {
        B.status[lp] = status;
        B.iters[lp] = iters;
        B.obj[lp] = T[(size_t)m * LD];
    }
}

__global__ void __launch_bounds__(kMaxThreads, 2)
fp64_resident_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                     int32_t* __restrict__ diag)
{
    extern __shared__ __align__(16) unsigned char smem[];
    solve_one(B, tol, order[blockIdx.x], smem, smem + SmallLayout::total, diag);
}

// One warp per LP (blockDim = 32), the form of the groups of small tableaux:
// the same per-LP code with warp barriers and `redux` reductions instead of
// block barriers and shared-memory round trips; the same arithmetic.
__global__ void __launch_bounds__(32, 32)
fp64_warp_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                 int32_t* __restrict__ diag)
{
    extern __shared__ __align__(16) unsigned char smem[];
    solve_one<true>(B, tol, order[blockIdx.x], smem, smem + SmallLayout::total, diag);
}

// Resident kernel over a device-side list: persistent CTAs take the LPs
// queue[0 .. *queue_len) through the atomic `counter` (0 at launch).  Used for
// the LPs the mixed-precision kernel hands back.
__global__ void __launch_bounds__(kMaxThreads, 2)
fp64_resident_queue_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ queue,
                           const int32_t* __restrict__ queue_len, const int32_t queue_cap, const int32_t num_lps,
                           int32_t* __restrict__ counter, int32_t* __restrict__ diag)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int next;
    const int count = min(*queue_len, queue_cap);
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        __syncthreads();
        const int idx = next;
        __syncthreads();
        if (idx >= count) break;
        const int lp = queue[idx];
        if (lp < 0 || lp >= num_lps) {
            if (threadIdx.x == 0) record_internal_error(diag, 5, lp);
            continue;
        }
        solve_one(B, tol, lp, smem, smem + SmallLayout::total, diag);
        __syncthreads();
    }
}


// One LP of any size with deferred updates: its vectors and first pending
// pivots in `bytes` of shared memory when the vectors fit (phase I's, at their
// largest), else in the workspace slot.
__device__ __forceinline__ void deferred_large(const DeviceBatch& B, const Tolerances& tol, const int lp,
                                               unsigned char* small, unsigned char* shared, const size_t bytes,
                                               unsigned char* slot, int32_t* diag)
{
    DeferBlock g(small);
    if (deferred_layout(B.m[lp], B.n[lp], B.m[lp]).hist <= bytes)
        deferred_solve_large(g, B, tol, lp, shared, bytes, slot, diag);
    else
        deferred_solve_large(g, B, tol, lp, slot, 0, slot, diag);
}

// LPs whose tableau is not kept in shared memory (lp_fp64_deferred.cuh):
// persistent CTAs take them from the atomic `counter`; CTA i owns workspace
// slot i.  One warp per LP, one CTA per LP, and one CTA per LP of any size.
enum DeferredKind { kDeferOneWarp, kDeferCta, kDeferLarge };
template <DeferredKind kKind>
__device__ __forceinline__ void deferred_queue(const DeviceBatch& B, const Tolerances& tol,
                                               const int32_t* __restrict__ order, const int32_t count,
                                               const int32_t* __restrict__ count_dev, unsigned char* workspace,
                                               const size_t slot_bytes, int32_t* __restrict__ counter,
                                               int32_t* __restrict__ diag, const size_t smem_bytes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int next;
    unsigned char* slot = workspace + (size_t)blockIdx.x * slot_bytes;
    const int n_items = count_dev ? min(*count_dev, count) : count;
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        __syncthreads();
        const int idx = next;
        __syncthreads();
        if (idx >= n_items) break;
        const int lp = order[idx];
        if constexpr (kKind == kDeferOneWarp) {
            DeferWarp g;
            deferred_solve(g, B, tol, lp, smem, smem_bytes, slot, diag);
        } else if constexpr (kKind == kDeferCta) {
            DeferBlock g(smem);
            deferred_solve(g, B, tol, lp, smem + SmallLayout::total, smem_bytes - SmallLayout::total, slot, diag);
        } else {
            deferred_large(B, tol, lp, smem, smem + SmallLayout::total, smem_bytes - SmallLayout::total, slot, diag);
        }
        __syncthreads();
    }
}

__global__ void __maxnreg__(80)
fp64_deferred_warp_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                          const int32_t count, const int32_t* __restrict__ count_dev, unsigned char* workspace,
                          const size_t slot_bytes, int32_t* __restrict__ counter, int32_t* __restrict__ diag,
                          const size_t smem_bytes)
{
    deferred_queue<kDeferOneWarp>(B, tol, order, count, count_dev, workspace, slot_bytes, counter, diag, smem_bytes);
}

__global__ void __maxnreg__(80)
fp64_deferred_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                     const int32_t count, const int32_t* __restrict__ count_dev, unsigned char* workspace,
                     const size_t slot_bytes, int32_t* __restrict__ counter, int32_t* __restrict__ diag,
                     const size_t smem_bytes)
{
    deferred_queue<kDeferCta>(B, tol, order, count, count_dev, workspace, slot_bytes, counter, diag, smem_bytes);
}

__global__ void __launch_bounds__(kMaxThreads, 2)
fp64_deferred_large_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                           const int32_t count, const int32_t* __restrict__ count_dev, unsigned char* workspace,
                           const size_t slot_bytes, int32_t* __restrict__ counter, int32_t* __restrict__ diag,
                           const size_t smem_bytes)
{
    deferred_queue<kDeferLarge>(B, tol, order, count, count_dev, workspace, slot_bytes, counter, diag, smem_bytes);
}

// A whole batch in one launch: persistent CTAs take the LPs order[0 ..
// count) (longest work first) from the atomic `counter` and solve each with
// the tableau in this CTA's shared memory when it fits (resident[lp] != 0),
// else with deferred updates and this CTA's global workspace slot -- the same
// per-LP code as the resident and deferred kernels, so the same results.
__global__ void __launch_bounds__(kSingleThreads, 2)
fp64_single_kernel(const DeviceBatch B, const Tolerances tol, const int32_t* __restrict__ order,
                   const uint8_t* __restrict__ resident, const int32_t count, unsigned char* workspace,
                   const size_t slot_bytes, int32_t* __restrict__ counter, int32_t* __restrict__ diag,
                   const size_t smem_bytes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int next;
    unsigned char* slot = workspace ? workspace + (size_t)blockIdx.x * slot_bytes : nullptr;
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(counter, 1);
        __syncthreads();
        const int idx = next;
        __syncthreads();
        if (idx >= count) break;
        const int lp = order[idx];
        if (resident[lp]) {
            solve_one(B, tol, lp, smem, smem + SmallLayout::total, diag);
        } else if (slot) {
            deferred_large(B, tol, lp, smem, smem + SmallLayout::total, smem_bytes - SmallLayout::total, slot, diag);
        } else if (threadIdx.x == 0) {
            record_internal_error(diag, 7, lp);  // a plan without a slot for an LP that needs one
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t fp64_kernels_prepare() {
    cudaError_t err = cudaFuncSetAttribute(fp64_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kMaxSmemPerBlock);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(fp64_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmemPerBlock);
    if (err != cudaSuccess) return err;
    return cudaFuncSetAttribute(fp64_resident_queue_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(kMaxSmemPerBlock - 1024));
}

int fp64_resident_queue_ctas_per_sm(int threads, size_t smem) {
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fp64_resident_queue_kernel, threads, smem) != cudaSuccess)
        return 1;
    return blocks > 0 ? blocks : 1;
}

cudaError_t launch_fp64_resident_queue(const DeviceBatch& B, const Tolerances& tol, const int32_t* queue,
                                       const int32_t* queue_len, int32_t queue_cap, int32_t num_lps,
                                       int32_t* counter, int32_t* diag, int ctas, int threads,
                                       size_t smem, cudaStream_t stream) {
    cudaError_t err = cudaMemsetAsync(counter, 0, sizeof(int32_t), stream);
    if (err != cudaSuccess) return err;
    fp64_resident_queue_kernel<<<ctas, threads, smem, stream>>>(B, tol, queue, queue_len, queue_cap, num_lps,
                                                                counter, diag);
    return cudaGetLastError();
}

// Deferred updates for every tableau above one CTA's shared memory, and below
// that by size, shape and sign.  They save FMAs while few pivots are pending, and
// spread a pivot's work over fewer threads; an LP that has to flush makes them
// all after all.  The number of pivots decides, and is not known beforehand.
// Measured on 1000 LPs, deferred / resident, ms:
//  - packing LPs (no negative entry in A: few pivots) of both sides >= 32: 45 x 45
//    (20,000) 0.47 / 0.74, 80 x 80 (2400) 0.28 / 0.39, 130 x 130 0.19 / 0.67, but 30 x 70
//    0.54 / 0.50 and 16 x 130 0.97 / 0.56 (the pivot's fixed cost counts);
//  - packing LPs of a shorter side, above 14,000 entries: 16 x 900 0.95 / 1.07, 24 x 600
//    0.77 / 0.90, 750 x 20 0.24 / 0.61, 1600 x 8 0.31 / 0.72; with rows of more than 1024
//    entries, which only one CTA per SM has room for, 8 x 1600 1.65 / 1.22, 12 x 1200
//    1.42 / 1.15, 20 x 1100 1.67 / 1.44;
//  - others, above 14,000 entries: rows longer than columns by half, 16 x 900 0.51 /
//    0.66, 24 x 1000 1.13 / 1.32, 64 x 225 2.3 / 2.5, 90 x 250 4.9 / 5.4, 120 x 180 9.4 /
//    9.9; a thread per row and column within 128, 125 x 125 13.1 / 13.8; fewer than 12
//    columns (no more pivots than are kept pending), 1450 x 10 0.84 / 1.01, 2000 x 6 0.68 /
//    0.85; but 130 x 130 17.0 / 15.5, with phase I 120 x 118 21.2 / 19.6, 300 x 48 4.5 / 3.8,
//    500 x 48 6.9 / 5.7, 1100 x 12 1.14 / 0.98, 16 x 1400 0.95 / 0.95 (with phase I 1.77 /
//    1.61); 225 x 64 4.9 / 5.6 and 160 x 90 8.6 / 9.1 are on the other side of the line.
bool defer_updates(int m, int n, int k, bool nonneg) {
    if (resident_smem_bytes(m, n, k) > kMaxSmemPerBlock) return true;
    const int w = n + k + 1, d = m > w ? m : w;
    const int64_t e = (int64_t)(m + 1) * w;
    if (nonneg && e > kDeferNonneg && m >= 32 && n >= 32) return true;
    if (e <= kDeferEntries) return false;
    if (d > 1024) return m > w && (nonneg || n < 12);
    return nonneg || d <= 128 || 2 * w >= 3 * m;
}

int resident_threads(int m, int n, int k) {
    const int64_t e = (int64_t)(m + 1 + (k > 0)) * (n + k + 1);
    // measured best on GB300 (mixed-sign dense m x m, m = 20..100)
    if (e <= 1024) return 32;
    if (e <= 3072) return 64;
    if (e <= 8192) return 128;
    if (e <= 32768) return 256;
    return 512;
}

// Size classes by the longer of a row and a column, d: a thread for each up to
// 256 (a warp's FP64 instruction holds its quarter of the SM's FP64 pipe for 64
// clocks, so one LP needs its elements spread over warps), 9 KB of shared memory
// per warp, 24 warps per SM at 80 registers.  Above, several per thread: 512
// threads; 256 and three CTAs per SM (class 4) only for packing LPs by the
// thousand (kDeferClass4PerSm), where throughput counts and not one LP's time.
// Class 4 / 5, ms: uneven packing LPs, 20,000 (4200 of class 4) 2.66 / 2.95, 10,000
// 1.73 / 1.71, 1000 0.92 / 0.75; 10,000 of 300 x 300 4.5 / 4.8, 2400 1.29 / 1.26, 200 0.35 /
// 0.25; with A in [1, 10] (43 pivots) 200 6.3 / 4.4 (5.1 with the whole tableau
// rewritten in the workspace at every pivot), 2400 9.3 / 7.4; 300 mixed-sign 300 x 300
// LPs 238 / 179.
DeferredForm deferred_class(int cls) {
    if (cls < 4) return {cls, 32 << cls, (size_t)(9 << 10) << cls};
    if (cls == 4) return {4, 256, 74 << 10};
    if (cls == 5) return {5, 512, 100 << 10};
    return {6, kMaxThreads, kMaxSmemPerBlock - 1024};
}

DeferredForm deferred_form(int m, int n, int k, bool nonneg) {
    const int d = m > n + k + 1 ? m : n + k + 1;
    for (int c = 0; c < 4; ++c)
        if (d <= (32 << c)) return deferred_class(c);
    if (d <= 1024) return deferred_class(nonneg && m >= 32 && n >= 32 ? 4 : 5);
    return deferred_class(6);
}

namespace {
using DeferredKernel = void (*)(const DeviceBatch, const Tolerances, const int32_t*, const int32_t, const int32_t*,
                                unsigned char*, const size_t, int32_t*, int32_t*, const size_t);
DeferredKernel deferred_kernel(const DeferredForm& f) {
    return f.cls == 0 ? fp64_deferred_warp_kernel : (f.cls < 4 ? fp64_deferred_kernel : fp64_deferred_large_kernel);
}
}  // namespace

int fp64_deferred_ctas_per_sm(const DeferredForm& f) {
    int blocks = 0;
    if (cudaFuncSetAttribute(deferred_kernel(f), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kMaxSmemPerBlock - 1024)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, deferred_kernel(f), f.threads, f.smem) != cudaSuccess)
        return 1;
    return blocks > 0 ? blocks : 1;
}

cudaError_t launch_fp64_deferred(const DeviceBatch& B, const Tolerances& tol, const int32_t* order, int32_t count,
                                 const DeferredForm& f, int slots, unsigned char* workspace, size_t slot_bytes,
                                 int32_t* counter, int32_t* diag, cudaStream_t stream, const int32_t* count_dev) {
    if (count <= 0) return cudaSuccess;
    cudaError_t err = cudaMemsetAsync(counter, 0, sizeof(int32_t), stream);
    if (err != cudaSuccess) return err;
    if ((err = cudaFuncSetAttribute(deferred_kernel(f), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kMaxSmemPerBlock - 1024))) != cudaSuccess)
        return err;
    deferred_kernel(f)<<<slots, f.threads, f.smem, stream>>>(B, tol, order, count, count_dev, workspace, slot_bytes,
                                                             counter, diag, f.smem);
    return cudaGetLastError();
}

// fp64_single_kernel: the largest dynamic shared memory that still lets
// `per_sm` CTAs share an SM, and how many do at a given size.
cudaError_t fp64_single_prepare(size_t smem) {
    return cudaFuncSetAttribute(fp64_single_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

int fp64_single_ctas_per_sm(size_t smem) {
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fp64_single_kernel, kSingleThreads, smem) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return blocks;
}

cudaError_t launch_fp64_single(const DeviceBatch& B, const Tolerances& tol, const int32_t* order,
                               const uint8_t* resident, int32_t count, int ctas, size_t smem,
                               unsigned char* workspace, size_t slot_bytes, int32_t* counter, int32_t* diag,
                               cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    cudaError_t err = cudaMemsetAsync(counter, 0, sizeof(int32_t), stream);
    if (err != cudaSuccess) return err;
    fp64_single_kernel<<<ctas, kSingleThreads, smem, stream>>>(B, tol, order, resident, count, workspace,
                                                                  slot_bytes, counter, diag, smem);
    return cudaGetLastError();
}

cudaError_t launch_fp64_resident(const DeviceBatch& B, const Tolerances& tol, const int32_t* order,
                                 int32_t count, int threads, size_t smem, int32_t* diag, cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    if (threads == 32)
        fp64_warp_kernel<<<count, 32, smem, stream>>>(B, tol, order, diag);
    else
        fp64_resident_kernel<<<count, threads, smem, stream>>>(B, tol, order, diag);
    return cudaGetLastError();
}

}  // namespace lpb
