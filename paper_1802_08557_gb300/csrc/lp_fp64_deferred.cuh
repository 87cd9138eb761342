// lp_fp64_deferred.cuh -- FP64 simplex of one LP with deferred updates: the
// per-LP code of the kernels whose tableau is not in shared memory
// (lp_fp64_simplex.cu).
//
// The rank-1 update of Step 3 (Gurung & Ray, arXiv 1802.08557, Section 3.1)
// rewrites every tableau element at every pivot, but a pivot only reads the
// objective row, the right-hand side, the entering column and the leaving row.
// Here the first two are updated at every pivot, and the body is not: pivot s
// leaves its column c_s (before the pivot) and its scaled row r_s in a
// history, and an element is formed when it is read, from its source value
// and the pending pivots in order,
//     t_ij <- fma(-c_s[i], r_s[j], t_ij)        s = 0, 1, ...
// -- the same operations in the same order as an update of the whole tableau
// makes on that element, so the results are the same bit for bit.  A row that
// was a pivot row restarts from r_s[j], a column that was the entering one
// from fma(-c_s[i], r_s[j], 0).  The source is the LP's A itself (no tableau
// is built).  When `first` pivots are pending the body is formed once in the
// LP's workspace slot (flush), which becomes the source.
//
// What it saves: t pending pivots cost t (m + n) FMAs per pivot instead of
// m n, and an LP of few pivots never touches most of its tableau.  On the FP64
// pipe of GB300 (2 lanes per SM and clock) the update was the whole cost: 20,000
// uneven LPs of 10-500 rows and columns, 8.5 pivots on average, need 3.9e8
// FMAs this way and 4.5e9 the other.  For long runs of pivots the flushes
// make the same FMAs per element as before but one pass over the tableau
// per `later` pivots, so the pass is bound by the FP64 pipe, not by memory.
//
// History: the first `ks` pending pivots in shared memory, the others in the
// slot (read in L2).  Every thread owns the rows i and the columns j congruent
// to its index; the barriers of one pivot are those of the two argmin
// exchanges and of the tie vote (3).  Two forms of the same arithmetic:
// deferred_solve, one row and one column per thread, in registers (one warp
// per LP up to 32 rows and columns); deferred_solve_large, several per thread,
// in memory, for any size.
#pragma once

#include "lp_device.cuh"
#include "lp_internal.h"

namespace lpb {
namespace {

// Exchange of per-warp results over the CTA through two alternating sets of
// slots: one barrier per exchange (a set is written again only after the next
// exchange's barrier, which every reader of it has passed).
struct Exchange {
    long long* k64;  // 2 x kMaxWarps
    unsigned* u32;   // 2 x 2 x kMaxWarps
    int nw, warp, lane;
    unsigned set;
    __device__ Exchange(unsigned char* small)
        : k64(reinterpret_cast<long long*>(small + SmallLayout::red64)),
          u32(reinterpret_cast<unsigned*>(small + SmallLayout::red32)), nw((int)(blockDim.x >> 5)),
          warp((int)(threadIdx.x >> 5)), lane((int)(threadIdx.x & 31)), set(0) {}

    // Lexicographic minimum of (key, sel) over the CTA and the OR of `flag`.
    __device__ void min_pair(long long& key, unsigned& sel, bool& flag) {
        long long km = warp_min_i64(key);
        unsigned sm = __reduce_min_sync(kFull, key == km ? sel : 0xffffffffu);
        const bool f = __any_sync(kFull, flag);
        set ^= 1u;
        long long* k = k64 + set * kMaxWarps;
        unsigned* s = u32 + set * 2 * kMaxWarps;
        if (lane == 0) {
            k[warp] = km;
            s[warp] = sm;
            s[kMaxWarps + warp] = f ? 1u : 0u;
        }
        __syncthreads();
        const bool in = lane < nw;
        const long long kl = in ? k[lane] : LLONG_MAX;
        const unsigned sl = in ? s[lane] : 0xffffffffu;
        flag = __any_sync(kFull, in && s[kMaxWarps + lane] != 0u);
        key = warp_min_i64(kl);
        sel = __reduce_min_sync(kFull, kl == key ? sl : 0xffffffffu);
    }
    __device__ long long min_i64(long long v) {
        unsigned s = 0;
        bool f = false;
        min_pair(v, s, f);
        return v;
    }
    __device__ unsigned min_u32(unsigned v) {
        v = __reduce_min_sync(kFull, v);
        set ^= 1u;
        unsigned* s = u32 + set * 2 * kMaxWarps;
        if (lane == 0) s[warp] = v;
        __syncthreads();
        return __reduce_min_sync(kFull, lane < nw ? s[lane] : 0xffffffffu);
    }
    // Exclusive prefix count of `flag` in thread order, and the total.
    __device__ int prefix_count(bool flag, int& total) {
        const unsigned bal = __ballot_sync(kFull, flag);
        set ^= 1u;
        unsigned* s = u32 + set * 2 * kMaxWarps;
        if (lane == 0) s[warp] = (unsigned)__popc(bal);
        __syncthreads();
        const unsigned c = lane < nw ? s[lane] : 0u;
        total = (int)__reduce_add_sync(kFull, c);
        return (int)__reduce_add_sync(kFull, lane < warp ? c : 0u) + __popc(bal & ((1u << lane) - 1u));
    }
};

// v <- fma(-b_s, y_s, v) for s = max(from, s0) .. to-1, with b_s = bp[s * bs]
// and y_s = vp[s * vs].  (-c) r and (-r) c are the same product, so this
// serves columns (b = r_s[e], y = c_s[i]) and rows (b = c_s[l], y = r_s[j])
// alike.  One element per lane and step: a warp's FP64 instruction keeps its
// part of the FP64 pipe busy for longer than the FMA's latency, so several
// chains per lane gained nothing and cost instruction cache.
__device__ __forceinline__ double chain(double v, int s0, int from, int to, const double* bp, int bs,
                                        const double* vp, int vs) {
    bp += (ptrdiff_t)from * bs;
    vp += (ptrdiff_t)from * vs;
#pragma unroll 4
    for (int s = from; s < to; ++s) {
        const double b = -*bp, y = *vp;
        if (s >= s0) v = __fma_rn(b, y, v);
        bp += bs;
        vp += vs;
    }
    return v;
}

// The group of threads that owns an LP: a CTA (exchanges through shared memory,
// every call a barrier) or one warp (redux only).
struct DeferBlock : Exchange {
    int tid, nt;
    __device__ explicit DeferBlock(unsigned char* small)
        : Exchange(small), tid((int)threadIdx.x), nt((int)blockDim.x) {}
    __device__ void sync() { __syncthreads(); }
    __device__ bool any(bool v) { return __syncthreads_or(v) != 0; }
};
struct DeferWarp {
    int tid, nt, nw, warp, lane;
    __device__ DeferWarp()
        : tid((int)(threadIdx.x & 31)), nt(32), nw(1), warp(0), lane((int)(threadIdx.x & 31)) {}
    __device__ void sync() { __syncwarp(); }
    __device__ bool any(bool v) {
        __syncwarp();
        return __any_sync(kFull, v) != 0;
    }
    __device__ void min_pair(long long& key, unsigned& sel, bool& flag) {
        __syncwarp();
        const long long km = warp_min_i64(key);
        sel = __reduce_min_sync(kFull, key == km ? sel : 0xffffffffu);
        key = km;
        flag = __any_sync(kFull, flag) != 0;
    }
    __device__ long long min_i64(long long v) {
        __syncwarp();
        return warp_min_i64(v);
    }
    __device__ unsigned min_u32(unsigned v) {
        __syncwarp();
        return __reduce_min_sync(kFull, v);
    }
    __device__ int prefix_count(bool flag, int& total) {
        __syncwarp();
        const unsigned bal = __ballot_sync(kFull, flag);
        total = __popc(bal);
        return __popc(bal & ((1u << lane) - 1u));
    }
};

// One LP, Steps 1-3 until it halts, by the group g of at least max(m, n + k + 1)
// threads: thread t owns row t and column t, in registers.  In `base`
// (`base_bytes` of shared memory): what owners tell the others, and the first
// pending pivots; the body and the other pending pivots in `slot`
// (DeferredSlot).
template <class G>
__device__ __forceinline__ void deferred_solve(G& g, const DeviceBatch& B, const Tolerances& tol, const int lp,
                                               unsigned char* base, const size_t base_bytes, unsigned char* slot,
                                               int32_t* diag)
{
    const int m = B.m[lp];
    const int n = B.n[lp];
    const int nm = n + m;
    const double* __restrict__ A = B.A + B.a_off[lp];
    const double* __restrict__ bv = B.b + B.b_off[lp];
    const double* __restrict__ cv = B.c + B.c_off[lp];
    const int tid = g.tid;
    const DeferredRegLayout L0 = deferred_reg_layout(m, n, 0);
    // box: objective entries of the entering column (0, 1), the leaving row's
    // right-hand side (2); boxi: its basic variable, restart point and sign
    double* box = reinterpret_cast<double*>(base + L0.box);
    int* boxi = reinterpret_cast<int*>(base + L0.box + 32);
    unsigned* negbits = reinterpret_cast<unsigned*>(base + L0.negbits);  // negated rows
    int* neg = reinterpret_cast<int*>(base + L0.neg);                    // ... as an ascending list
    int* row_last = reinterpret_cast<int*>(base + L0.row_last);          // (copies, for the flush
    int* col_last = reinterpret_cast<int*>(base + L0.col_last);          //  and a column's start)
    auto too_big = [&](int k) {
        if (tid == 0) {
            record_internal_error(diag, 10, lp, m, n, k);
            B.status[lp] = kNumerical;
        }
    };
    if (m > g.nt || n >= g.nt || L0.hist > base_bytes) return too_big(0);

    // rows with b_i < 0 are negated and get an artificial (two-phase method, Section 3)
    const bool has_row = tid < m;
    const double b0 = has_row ? bv[tid] : 0.0;
    const bool negated = b0 < 0.0;
    int k;
    const int rank = g.prefix_count(negated, k);
    const unsigned bal = __ballot_sync(kFull, negated);
    if (g.lane == 0 && has_row) negbits[tid >> 5] = bal;
    if (negated) neg[rank] = tid;
    if (has_row) row_last[tid] = -1;
    double beta = negated ? -b0 : b0, vcol = 0.0;               // right-hand side; entry of the last pivot's column
    int rvar = negated ? nm + rank : n + tid, rlast = -1;       // basic variable; last pending pivot on the row
    const long long bmax_key = -g.min_i64(-max(0x3FF0000000000000LL, abskey(b0)));  // also orders neg[], negbits[]
    const int W = n + k + 1;  // columns: 0 the right-hand side, 1.. the non-basic variables
    const DeferredRegLayout L = deferred_reg_layout(m, n, k);
    if (W > g.nt || L.hist > base_bytes) return too_big(k);
    const DeferredSlot S = deferred_slot(m, n, k);
    double* T = reinterpret_cast<double*>(slot + S.T);
    const int LD = S.LD;
    // pending pivots [0, ks) in `base`, the others in the slot
    const int ks = (int)min((size_t)S.first, (base_bytes - L.hist) / ((size_t)(m + W) * 8));
    double* cs = reinterpret_cast<double*>(base + L.hist);  // c_s at cs + s * m
    double* rs = cs + (size_t)ks * m;                       // r_s at rs + s * W
    double* cg = reinterpret_cast<double*>(slot + S.hist) - (ptrdiff_t)ks * m;
    double* rg = reinterpret_cast<double*>(slot + S.hist) + (size_t)S.first * m - (ptrdiff_t)ks * W;
    int cap = S.first;  // pending pivots before the next flush

    constexpr int kRetired = INT_MAX;  // col_last of a retired column
    bool from_a = true;  // the source of an element: A, or T after a flush
    auto source = [&](int i, int j, bool neg_i) -> double {  // j >= 1
        if (!from_a) return T[(size_t)i * LD + j];
        const double v = (j <= n) ? A[(size_t)i * n + j - 1] : ((neg[j - 1 - n] == i) ? 1.0 : 0.0);
        return neg_i ? -v : v;
    };
    // own column: variable (nm and above: retired, column 0 or none), last
    // pending pivot on it, objective row(s)
    const bool has_col = tid < W;
    int cvar = INT_MAX, clast = -1;
    double obj = 0.0, aux = 0.0;
    if (has_col) {
        col_last[tid] = -1;
        if (tid >= 1) cvar = tid <= n ? tid - 1 : n + neg[tid - 1 - n];
        if (tid >= 1 && tid <= n) obj = -cv[tid - 1];
        // auxiliary objective: maximise -(sum of artificials), priced out by
        // subtracting every negated row in ascending row order
#pragma unroll 4
        for (int u = 0; u < k; ++u) aux = __dsub_rn(aux, tid == 0 ? -bv[neg[u]] : source(neg[u], tid, true));
    }

    const long long key_neg_eps_opt = okey(-tol.eps_opt);
    const long long key_eps_piv = okey(tol.eps_piv);
    const int max_iters = tol.max_iters > 0 ? tol.max_iters : 50 * (m + n);
    int iters = 0, status = -1;
    bool one = k > 0, infeasible = false;  // one: phase I
    int t = 0;         // pending pivots
    int rhs_row = -1;  // pivot row of pivot t-1 while the right-hand side waits for it, else -1

    auto c_at = [&](int s) { return s < ks ? cs + (size_t)s * m : cg + (ptrdiff_t)s * m; };
    auto r_at = [&](int s) { return s < ks ? rs + (size_t)s * W : rg + (ptrdiff_t)s * W; };
    // beta <- the right-hand side after pivot t-1 (after a barrier that follows it)
    auto settle_rhs = [&]() {
        if (rhs_row < 0) return;
        if (has_row) {
            const double q0 = r_at(t - 1)[0];
            beta = (tid == rhs_row) ? q0 : __fma_rn(-vcol, q0, beta);
        }
        rhs_row = -1;
    };
    // start of element (i, j)'s chain: its value and its first pivot
    auto begin = [&](int i, int j, int sr, int sc, bool neg_i, int& s0) -> double {
        const int last = max(sr, sc);
        s0 = last + 1;
        if (last < 0) return source(i, j, neg_i);
        const double r = r_at(last)[j];
        return sr >= sc ? r : __fma_rn(-c_at(last)[i], r, 0.0);
    };
    // column e into vcol and c_at(t)
    auto column = [&](int e) {
        if (!has_row) return;
        const int sc = col_last[e];
        int s0;
        double v = begin(tid, e, rlast, sc, negated, s0);
        v = chain(v, s0, sc + 1, min(t, ks), rs + e, W, cs + tid, m);
        if (t > ks) v = chain(v, s0, max(sc + 1, ks), t, rg + e, W, cg + tid, m);
        vcol = v;
        c_at(t)[tid] = v;
    };
    // element (i, j) of a live column
    auto element = [&](int i, int j, int sr, int sc, bool neg_i) -> double {
        int s0;
        double v = begin(i, j, sr, sc, neg_i, s0);
        v = chain(v, s0, sr + 1, min(t, ks), cs + i, m, rs + j, W);
        if (t > ks) v = chain(v, s0, max(sr + 1, ks), t, cg + i, m, rg + j, W);
        return v;
    };
    // the body after every pending pivot, into T (the source from then on).  As
    // many threads per column as the group has, an element always by the same
    // thread: with one per column, LPs of few columns left most of the group idle.
    // 1000 signed LPs of 225 x 64 8.1 -> 4.9 ms, of 200 x 40 3.0 -> 1.5; without
    // allocation (a form for every row negated) 1500 of 200 x 40 8.6 -> 3.2, of 100 x
    // 100 10.8 -> 9.0.
    auto flush = [&]() {
        const int parts = g.nt / (W - 1), part = tid / (W - 1), j = 1 + tid - part * (W - 1);
        const int sc = part < parts ? col_last[j] : kRetired;
        if (sc != kRetired)
            for (int i = part; i < m; i += parts)
                T[(size_t)i * LD + j] = element(i, j, row_last[i], sc, (negbits[i >> 5] >> (i & 31)) & 1u);
        g.sync();
        rlast = clast = -1;
        if (has_row) row_last[tid] = -1;
        if (has_col && col_last[tid] != kRetired) col_last[tid] = -1;
        from_a = false;
        t = 0;
        cap = S.later;
        g.sync();
    };
    // Step 3's row: r_t, and the objective row(s) after the pivot.  u: the
    // unscaled own element; de, dw: objective entries of column e.
    auto scale = [&](double u, int e, double pe, double de, double dw, bool both) {
        if (tid != 0 && cvar >= nm) return;
        const bool at_e = tid == e;
        const double p = pivot_divide(at_e ? 1.0 : u, pe);
        r_at(t)[tid] = p;
        obj = __fma_rn(-de, p, at_e ? 0.0 : obj);
        if (both) aux = __fma_rn(-dw, p, at_e ? 0.0 : aux);
    };
    // labels and restart points of pivot t on (l, e), by their owners
    auto relabel = [&](int l, int e, int entering, int left) {
        if (tid == e) {
            cvar = left;  // an artificial (>= nm) retires with its column
            clast = t;
            col_last[e] = left < nm ? t : kRetired;
        }
        if (tid == l) {
            rvar = entering;
            rlast = row_last[l] = t;
        }
    };
    auto tell_row = [&](int l) {
        if (tid == l) {
            box[2] = beta;
            boxi[0] = rvar;
            boxi[1] = rlast;
            boxi[2] = negated ? 1 : 0;
        }
    };
    auto tell_objective = [&](int e) {
        if (tid == e) {
            box[0] = obj;
            box[1] = aux;
        }
    };
    const unsigned none = 0xffffffffu;

    while (status < 0) {
        // ---- Step 1: entering variable (most negative reduced cost) -------
        const bool live = cvar < nm;
        const unsigned mine = live ? ((unsigned)cvar << 16) | (unsigned)tid : none;
        const long long dkey = live ? okey(one ? aux : obj) : LLONG_MAX;
        long long dmin = dkey;
        unsigned esel = mine;
        bool others = false;
        g.min_pair(dmin, esel, others);
        settle_rhs();
        if (dmin >= key_neg_eps_opt) {
            if (!one) { status = kOptimal; break; }
            // ---- end of phase I (Section 3, two-phase method) -------------
            if (tid == 0) box[1] = aux;
            g.sync();
            if (-box[1] > __dmul_rn(tol.eps_feas, __longlong_as_double(bmax_key))) {
                status = kInfeasible;
                infeasible = true;
                break;
            }
            // drive artificials still basic (at level 0) out of the basis, in
            // ascending row order, on the lowest non-artificial column with |t_ij| > eps_piv
            for (int last = -1; status < 0;) {
                const unsigned next = g.min_u32(has_row && tid > last && rvar >= nm ? (unsigned)tid : none);
                if (next == none) break;
                const int i = last = (int)next;
                if (t == cap) flush();
                if (tid == i) {
                    box[2] = beta;
                    boxi[0] = rvar;
                    boxi[1] = rlast;
                    boxi[2] = negated ? 1 : 0;
                }
                g.sync();
                const double rhs = box[2];
                const int left = boxi[0];
                double u = rhs;
                unsigned sel = none;
                if (cvar < nm) {
                    u = element(i, tid, boxi[1], clast, boxi[2] != 0);
                    if (abskey(u) > key_eps_piv) sel = ((unsigned)cvar << 16) | (unsigned)tid;
                }
                sel = g.min_u32(sel);
                if (sel == none) continue;  // redundant row
                if (iters >= max_iters) { status = kIterLimit; break; }
                const int e = (int)(sel & 0xffffu);
                tell_objective(e);
                column(e);
                g.sync();
                scale(u, e, c_at(t)[i], box[0], 0.0, false);
                relabel(i, e, (int)(sel >> 16), left);
                ++t;
                ++iters;
                rhs_row = i;
                g.sync();
                settle_rhs();
            }
            one = false;
            continue;
        }
        if (t == cap) flush();
        // columns other than the minimum's within the tie-window bound of it
        // (see step1_window): told to the others with Step 2's exchange
        int e = (int)(esel & 0xffffu);
        others = live && tid != e &&
                 (unsigned long long)dkey - (unsigned long long)dmin <= step1_window(dmin, tol.key_window);

        // ---- Step 2: leaving row (minimum ratio rhs_i / t_ie, t_ie > eps) --
        // FP32 screen as in the shared-memory kernel: rows whose operands leave
        // [2^-100, 2^100] are always candidates (code INT_MIN)
        int code;
        long long rmin;
        unsigned lsel;
        for (bool again = false;;) {
            tell_objective(e);
            column(e);
            code = INT_MAX;  // not eligible
            if (has_row && okey(vcol) > key_eps_piv) {
                const int et = dexp(vcol), eb = dexp(beta);
                const bool safe = et >= -100 && et <= 100 && (abskey(beta) == 0 || (eb >= -100 && eb <= 100));
                code = safe ? fkey(__fdividef(f64_to_f32_trunc(beta), f64_to_f32_trunc(vcol))) : INT_MIN;
            }
            const bool screened = code != INT_MAX && code != INT_MIN;
            rmin = screened ? code : LLONG_MAX;
            lsel = screened ? (unsigned)tid : none;
            g.min_pair(rmin, lsel, others);
            if (again || !others) break;
            // several columns: the exact rule (lowest label within the window)
            const long long kthr = okey(tie_threshold(kval(dmin), tol.tau));
            esel = g.min_u32(live && dkey <= kthr ? mine : none);
            if ((int)(esel & 0xffffu) == e) break;
            e = (int)(esel & 0xffffu);
            again = true;
        }
        int fwin = INT_MIN, l = -1;
        if (lsel != none) {
            const float fm = fval((int)rmin);
            fwin = fkey(fm + __fmaf_rn(tol.ratio_rel, fabsf(fm), tol.ratio_abs));
            l = (int)lsel;
            tell_row(l);
        }
        const bool candidate = code == INT_MIN || (code != INT_MAX && code <= fwin);
        if (g.any(candidate && tid != l)) {
            // several rows: exact ratios of the candidates, exact rule
            const long long rk = candidate ? okey(__ddiv_rn(beta, vcol)) : LLONG_MAX;
            const long long kmin = g.min_i64(rk);
            const long long rthr = okey(tie_threshold(kval(kmin), tol.tau));
            l = (int)g.min_u32(has_row && rk <= rthr ? (unsigned)tid : none);
            if ((unsigned)l >= (unsigned)m) { status = kNumerical; break; }
            tell_row(l);
            g.sync();
        } else if (l < 0) {
            status = one ? kNumerical : kUnbounded;
            break;
        }
        const double pe = c_at(t)[l];
        if (abskey(pe) >= 0x7FF0000000000000LL) { status = kNumerical; break; }
        if (iters >= max_iters) { status = kIterLimit; break; }

        // ---- Step 3: pivot ---------------------------------------------------
        const int left = boxi[0];
        double u = box[2];
        if (live) u = element(l, tid, boxi[1], clast, boxi[2] != 0);
        scale(u, e, pe, box[0], box[1], one);
        relabel(l, e, (int)(esel >> 16), left);
        rhs_row = l;
        ++t;
        ++iters;
    }

    // ---- labels must name variables (self-check before they index global
    // memory); a failure is recorded and the LP reported as LP_NUMERICAL ----
    const unsigned nvar = (unsigned)(nm + k);
    const bool bad = (has_row && (unsigned)rvar >= nvar) || (has_col && tid >= 1 && (unsigned)cvar >= nvar);
    if (g.min_u32(bad ? 0u : 1u) == 0u) {
        if (tid == 0) {
            record_internal_error(diag, 6, lp, 0, status, iters, one ? 1 : 2, W);
            B.status[lp] = kNumerical;
            B.iters[lp] = iters;
        }
        return;
    }
    // ---- results: x (basic rows -> rhs, non-basic -> 0), y (slack reduced
    // costs of the last objective row), objective corner, status, pivots ------
    double* __restrict__ x = B.x + B.x_off[lp];
    double* __restrict__ y = B.y ? B.y + B.y_off[lp] : nullptr;
    if (cvar < n) x[cvar] = 0.0;
    else if (cvar < nm && y) y[cvar - n] = infeasible ? aux : obj;
    if (has_row) {
        if (rvar < n) x[rvar] = beta;
        else if (rvar < nm && y) y[rvar - n] = 0.0;
    }
    if (tid == 0) {
        B.status[lp] = status;
        B.iters[lp] = iters;
        B.obj[lp] = obj;
    }
}

// One LP of any size, by the CTA g.  The LP's vectors and the first pending
// pivots are in `base` (`base_bytes` of shared memory, or of the
// slot when the vectors alone exceed shared memory), the body and the other
// pending pivots in `slot` (DeferredSlot).
__device__ __forceinline__ void deferred_solve_large(DeferBlock& g, const DeviceBatch& B, const Tolerances& tol, const int lp,
                                                     unsigned char* base, const size_t base_bytes,
                                                     unsigned char* slot, int32_t* diag)
{
    const int m = B.m[lp];
    const int n = B.n[lp];
    const int nm = n + m;
    const double* __restrict__ A = B.A + B.a_off[lp];
    const double* __restrict__ bv = B.b + B.b_off[lp];
    const double* __restrict__ cv = B.c + B.c_off[lp];
    const int tid = g.tid, nt = g.nt, lane = g.lane, warp = g.warp, nw = g.nw;

    const DeferredLayout L0 = deferred_layout(m, n, 0);
    double* beta = reinterpret_cast<double*>(base + L0.beta);            // right-hand side
    int* code = reinterpret_cast<int*>(base + L0.code);                  // Step 2 ratio codes
    int* row_var = reinterpret_cast<int*>(base + L0.row_var);            // basic variable of each row
    int* row_last = reinterpret_cast<int*>(base + L0.row_last);          // last pending pivot on the row, or -1
    int* negidx = reinterpret_cast<int*>(base + L0.negidx);              // rank among the negated rows, or -1
    int* neg = reinterpret_cast<int*>(base + L0.neg);                    // negated rows in ascending order

    // rows with b_i < 0 are negated and get an artificial (two-phase method, Section 3)
    int k = 0;
    long long bmax_key = 0x3FF0000000000000LL;  // 1.0
    for (int i0 = 0; i0 < m; i0 += nt) {
        const int i = i0 + tid;
        const double bi = (i < m) ? bv[i] : 0.0;
        const bool isneg = bi < 0.0;
        int tot;
        const int r = k + g.prefix_count(isneg, tot);
        if (i < m) {
            if (isneg) neg[r] = i;
            negidx[i] = isneg ? r : -1;
            row_var[i] = isneg ? nm + r : n + i;
            row_last[i] = -1;
            beta[i] = isneg ? -bi : bi;
            bmax_key = max(bmax_key, abskey(bi));
        }
        k += tot;
    }
    bmax_key = -g.min_i64(-bmax_key);  // also orders neg[] and negidx[] before their readers below

    const DeferredLayout L = deferred_layout(m, n, k);
    const int W = n + k + 1;  // columns: 0 the right-hand side, 1.. the non-basic variables
    double* obj = reinterpret_cast<double*>(base + L.obj);
    double* aux = reinterpret_cast<double*>(base + L.aux);
    int* col_var = reinterpret_cast<int*>(base + L.col_var);    // variable of each column (>= nm: retired)
    int* col_last = reinterpret_cast<int*>(base + L.col_last);  // last pending pivot on the column, or -1
    const DeferredSlot S = deferred_slot(m, n, k);
    double* T = reinterpret_cast<double*>(slot + S.T);
    const int LD = S.LD;
    // history: pending pivots [0, ks) in `base`, the others in the slot
    const size_t per = (size_t)(m + W) * 8;
    const int ks = base_bytes > L.hist ? (int)min((size_t)S.first, (base_bytes - L.hist) / per) : 0;
    double* cs = reinterpret_cast<double*>(base + L.hist);  // c_s at cs + s * m
    double* rs = cs + (size_t)ks * m;                       // r_s at rs + s * W
    // (offset so that pivot s >= ks sits at cg + s * m, rg + s * W)
    double* cg = reinterpret_cast<double*>(slot + S.hist) - (ptrdiff_t)ks * m;
    double* rg = reinterpret_cast<double*>(slot + S.hist) + (size_t)S.first * m - (ptrdiff_t)ks * W;
    int cap = S.first;  // pending pivots before the next flush

    bool from_a = true;  // the source of an element: A, or T after a flush
    auto source = [&](int i, int j) -> double {
        if (!from_a) return T[(size_t)i * LD + j];
        const double v = (j <= n) ? A[(size_t)i * n + j - 1] : ((neg[j - 1 - n] == i) ? 1.0 : 0.0);
        return (negidx[i] >= 0) ? -v : v;
    };

    for (int j = tid; j < W; j += nt) {
        col_var[j] = (j == 0) ? -1 : (j <= n ? j - 1 : n + neg[j - 1 - n]);
        col_last[j] = -1;
        obj[j] = (j >= 1 && j <= n) ? -cv[j - 1] : 0.0;
        if (k > 0) {
            // auxiliary objective: maximise -(sum of artificials), priced out by
            // subtracting every negated row in ascending row order
            double w = 0.0;
#pragma unroll 4
            for (int t = 0; t < k; ++t) w = __dsub_rn(w, j == 0 ? -bv[neg[t]] : source(neg[t], j));
            aux[j] = w;
        }
    }

    const long long key_neg_eps_opt = okey(-tol.eps_opt);
    const long long key_eps_piv = okey(tol.eps_piv);
    const int max_iters = tol.max_iters > 0 ? tol.max_iters : 50 * (m + n);
    int iters = 0, status = -1, phase = (k > 0) ? 1 : 2;
    bool infeasible = false;
    int t = 0;             // pending pivots
    int rhs_row = -1;      // pivot row of pivot t-1 while the right-hand side waits for it, else -1

    auto c_at = [&](int s) { return s < ks ? cs + (size_t)s * m : cg + (ptrdiff_t)s * m; };
    auto r_at = [&](int s) { return s < ks ? rs + (size_t)s * W : rg + (ptrdiff_t)s * W; };

    // beta <- the right-hand side after pivot t-1 (after a barrier that follows it)
    auto settle_rhs = [&]() {
        if (rhs_row < 0) return;
        const double q0 = r_at(t - 1)[0];
        const double* c = c_at(t - 1);
        for (int i = tid; i < m; i += nt) beta[i] = (i == rhs_row) ? q0 : __fma_rn(-c[i], q0, beta[i]);
        rhs_row = -1;
    };
    // start of element (i, j)'s chain: its value and its first pivot
    auto begin = [&](int i, int j, int sr, int sc, int& s0) -> double {
        if (sr < 0 && sc < 0) {
            s0 = 0;
            return source(i, j);
        }
        if (sr >= sc) {
            s0 = sr + 1;
            return r_at(sr)[j];
        }
        s0 = sc + 1;
        return __fma_rn(-c_at(sc)[i], r_at(sc)[j], 0.0);
    };
    // column e into c_at(t); `each(i, value)` for every own row
    auto column = [&](int e, auto each) {
        const int sc = col_last[e];
        double* dst = c_at(t);
        for (int i = tid; i < m; i += nt) {
            int s0;
            double v = begin(i, e, row_last[i], sc, s0);
            v = chain(v, s0, sc + 1, min(t, ks), rs + e, W, cs + i, m);
            if (t > ks) v = chain(v, s0, max(sc + 1, ks), t, rg + e, W, cg + i, m);
            dst[i] = v;
            each(i, v);
        }
    };
    // row l, `each(j, value)` for the live columns j0, j0 + step, ... (j >= 1)
    auto row = [&](int l, int sr, int j0, int step, auto each) {
        for (int j = j0; j < W; j += step) {
            if (j < 1 || col_var[j] >= nm) continue;
            int s0;
            double v = begin(l, j, sr, col_last[j], s0);
            v = chain(v, s0, sr + 1, min(t, ks), cs + l, m, rs + j, W);
            if (t > ks) v = chain(v, s0, max(sr + 1, ks), t, cg + l, m, rg + j, W);
            each(j, v);
        }
    };
    // the body after every pending pivot, into T (the source from then on)
    auto flush = [&]() {
        for (int i = warp; i < m; i += nw) {
            double* Ti = T + (size_t)i * LD;
            row(i, row_last[i], 1 + lane, 32, [&](int j, double v) { Ti[j] = v; });
        }
        g.sync();
        for (int i = tid; i < m; i += nt) row_last[i] = -1;
        for (int j = tid; j < W; j += nt) col_last[j] = -1;
        from_a = false;
        t = 0;
        cap = S.later;
        g.sync();
    };
    // Step 3's row: r_t from the unscaled row values, and the objective row(s)
    // after the pivot (`both`: phase I's two).  de, dw: their entries of column e.
    auto scale = [&](int j, double u, int e, double pe, double de, double dw, bool both) {
        const double q = pivot_divide(j == e ? 1.0 : u, pe);
        r_at(t)[j] = q;
        obj[j] = __fma_rn(-de, q, j == e ? 0.0 : obj[j]);
        if (both) aux[j] = __fma_rn(-dw, q, j == e ? 0.0 : aux[j]);
    };
    // labels and restart points of pivot t on (l, e), by their owners
    auto relabel = [&](int l, int e, int entering, int left) {
        if (tid == e % nt) {
            col_var[e] = left;  // an artificial (>= nm) retires with its column
            col_last[e] = t;
        }
        if (tid == l % nt) {
            row_var[l] = entering;
            row_last[l] = t;
        }
    };

    while (status < 0) {
        const double* orow = (phase == 1) ? aux : obj;
        // ---- Step 1: entering variable (most negative reduced cost) -------
        // over the own columns, which this thread wrote itself: no barrier
        long long dmin = LLONG_MAX;
        unsigned esel = 0xffffffffu;
        for (int j = tid; j < W; j += nt) {
            const int v = col_var[j];
            if (j >= 1 && v < nm) {
                const long long kj = okey(orow[j]);
                const unsigned sj = ((unsigned)v << 16) | (unsigned)j;
                if (kj < dmin || (kj == dmin && sj < esel)) {
                    dmin = kj;
                    esel = sj;
                }
            }
        }
        bool others = false;
        g.min_pair(dmin, esel, others);
        settle_rhs();
        if (dmin >= key_neg_eps_opt) {
            if (phase == 2) { status = kOptimal; break; }
            // ---- end of phase I (Section 3, two-phase method) -------------
            if (-aux[0] > __dmul_rn(tol.eps_feas, __longlong_as_double(bmax_key))) {
                status = kInfeasible;
                infeasible = true;
                break;
            }
            // drive artificials still basic (at level 0) out of the basis on
            // the lowest non-artificial column with |t_ij| > eps_piv
            for (int i = 0; i < m && status < 0; ++i) {
                if (row_var[i] < nm) continue;
                if (t == cap) flush();
                unsigned sel = 0xffffffffu;
                double* rt = r_at(t);
                const int sr = row_last[i];
                row(i, sr, tid, nt, [&](int j, double u) {
                    rt[j] = u;
                    if (abskey(u) > key_eps_piv) sel = min(sel, ((unsigned)col_var[j] << 16) | (unsigned)j);
                });
                sel = g.min_u32(sel);
                if (sel == 0xffffffffu) continue;  // redundant row
                if (iters >= max_iters) { status = kIterLimit; break; }
                const int e = (int)(sel & 0xffffu);
                const double de = obj[e];
                const int left = row_var[i];
                column(e, [](int, double) {});
                g.sync();
                const double pe = c_at(t)[i];
                for (int j = tid; j < W; j += nt)
                    if (j == 0 || col_var[j] < nm) scale(j, j == 0 ? beta[i] : rt[j], e, pe, de, 0.0, false);
                relabel(i, e, (int)(sel >> 16), left);
                ++t;
                ++iters;
                rhs_row = i;
                g.sync();
                settle_rhs();
                g.sync();
            }
            phase = 2;
            continue;
        }
        if (t == cap) flush();
        // columns other than the minimum's within the tie-window bound of it
        // (see step1_window): told to the others with Step 2's exchange
        const unsigned long long win = step1_window(dmin, tol.key_window);
        int e = (int)(esel & 0xffffu);
        for (int j = tid; j < W; j += nt)
            others |= j >= 1 && j != e && col_var[j] < nm &&
                      (unsigned long long)okey(orow[j]) - (unsigned long long)dmin <= win;

        // ---- Step 2: leaving row (minimum ratio rhs_i / t_ie, t_ie > eps) --
        // FP32 screen as in the shared-memory kernel: rows whose operands leave
        // [2^-100, 2^100] are always candidates
        long long rmin;
        unsigned lsel;
        for (bool again = false;;) {
            rmin = LLONG_MAX;
            lsel = 0xffffffffu;
            column(e, [&](int i, double te) {
                int ci = INT_MAX;  // not eligible
                if (okey(te) > key_eps_piv) {
                    const double bi = beta[i];
                    const int et = dexp(te), eb = dexp(bi);
                    if (et >= -100 && et <= 100 && (abskey(bi) == 0 || (eb >= -100 && eb <= 100))) {
                        ci = fkey(__fdividef(f64_to_f32_trunc(bi), f64_to_f32_trunc(te)));
                        if (ci < rmin) {  // rows ascend: the first of equals stays
                            rmin = ci;
                            lsel = (unsigned)i;
                        }
                    } else {
                        ci = INT_MIN;  // unscreened
                    }
                }
                code[i] = ci;
            });
            g.min_pair(rmin, lsel, others);
            if (again || !others) break;
            // several columns: the exact rule (lowest label within the window)
            const long long kthr = okey(tie_threshold(kval(dmin), tol.tau));
            unsigned sel = 0xffffffffu;
            for (int j = tid; j < W; j += nt) {
                const int v = col_var[j];
                if (j >= 1 && v < nm && okey(orow[j]) <= kthr) sel = min(sel, ((unsigned)v << 16) | (unsigned)j);
            }
            esel = g.min_u32(sel);
            if ((int)(esel & 0xffffu) == e) break;
            e = (int)(esel & 0xffffu);
            again = true;
        }
        const bool screened = rmin != LLONG_MAX;
        int fwin = INT_MIN;
        if (screened) {
            const float fm = fval((int)rmin);
            fwin = fkey(fm + __fmaf_rn(tol.ratio_rel, fabsf(fm), tol.ratio_abs));
        }
        // what the pivot overwrites, read before the vote's barrier
        int l = (int)lsel, left = -1, sr = -1;
        if (screened) {
            left = row_var[l];
            sr = row_last[l];
        }
        const double de = obj[e], dw = (phase == 1) ? aux[e] : 0.0;
        bool more = false;
        for (int i = tid; i < m; i += nt) {
            const int ci = code[i];
            more |= i != l && (ci == INT_MIN || (ci != INT_MAX && ci <= fwin));
        }
        const bool vote = g.any(more);
        if (!screened && !vote) {
            status = (phase == 2) ? kUnbounded : kNumerical;
            break;
        }
        if (vote) {
            // several rows: exact ratios of the candidates, exact rule (the ratio
            // of a row is formed again for the second pass: a rare path)
            const double* ct = c_at(t);
            auto ratio_key = [&](int i) -> long long {
                const int ci = code[i];
                if (ci != INT_MIN && (ci == INT_MAX || ci > fwin)) return LLONG_MAX;
                return okey(__ddiv_rn(beta[i], ct[i]));
            };
            long long rloc = LLONG_MAX;
            for (int i = tid; i < m; i += nt) rloc = min(rloc, ratio_key(i));
            const long long kmin = g.min_i64(rloc);
            const long long rthr = okey(tie_threshold(kval(kmin), tol.tau));
            unsigned sel = 0xffffffffu;
            for (int i = tid; i < m; i += nt)
                if (ratio_key(i) <= rthr) sel = min(sel, (unsigned)i);
            l = (int)g.min_u32(sel);
            if ((unsigned)l >= (unsigned)m) { status = kNumerical; break; }
            left = row_var[l];
            sr = row_last[l];
            g.sync();  // both read before their owner rewrites them
        }
        const double pe = c_at(t)[l];
        if (abskey(pe) >= 0x7FF0000000000000LL) { status = kNumerical; break; }
        if (iters >= max_iters) { status = kIterLimit; break; }

        // ---- Step 3: pivot ---------------------------------------------------
        row(l, sr, tid, nt, [&](int j, double u) { scale(j, u, e, pe, de, dw, phase == 1); });
        if (tid == 0) scale(0, beta[l], e, pe, de, dw, phase == 1);
        relabel(l, e, (int)(esel >> 16), left);
        rhs_row = l;
        ++t;
        ++iters;
    }

    // ---- labels must name variables (self-check before they index global
    // memory); a failure is recorded and the LP reported as LP_NUMERICAL ----
    {
        unsigned good = 1;
        const unsigned nvar = (unsigned)(nm + k);
        for (int i = tid; i < m; i += nt) good = ((unsigned)row_var[i] >= nvar) ? 0u : good;
        for (int j = tid; j < W; j += nt)
            if (j >= 1) good = ((unsigned)col_var[j] >= nvar) ? 0u : good;
        if (g.min_u32(good) == 0u) {
            if (tid == 0) {
                record_internal_error(diag, 6, lp, 0, status, iters, phase, W);
                B.status[lp] = kNumerical;
                B.iters[lp] = iters;
            }
            return;
        }
    }
    // ---- results: x (basic rows -> rhs, non-basic -> 0), y (slack reduced
    // costs of the last objective row), objective corner, status, pivots ------
    double* __restrict__ x = B.x + B.x_off[lp];
    double* __restrict__ y = B.y ? B.y + B.y_off[lp] : nullptr;
    const double* Ty = infeasible ? aux : obj;
    for (int j = tid; j < W; j += nt) {
        const int v = col_var[j];
        if (j == 0 || v >= nm) continue;
        if (v < n) x[v] = 0.0;
        else if (y) y[v - n] = Ty[j];
    }
    for (int i = tid; i < m; i += nt) {
        const int v = row_var[i];
        if (v < n) x[v] = beta[i];
        else if (v < nm && y) y[v - n] = 0.0;
    }
    if (tid == 0) {
        B.status[lp] = status;
        B.iters[lp] = iters;
        B.obj[lp] = obj[0];
    }
}

}  // namespace
}  // namespace lpb
