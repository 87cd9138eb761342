// lp_mixed_deferred.cuh -- the FP32 simplex of the mixed-precision path with
// deferred updates, as lp_fp64_deferred.cuh does it in FP64: a pivot leaves
// its column and its scaled row in a history, and an element is formed when it
// is read, from A (rounded to FP32) and the pending pivots in order -- the
// FMAs that an update of the whole tableau makes on it, so the results are the
// same bit for bit.  The objective row(s) and the right-hand side are updated
// at every pivot.  At the end only the columns that the FP64 certificate reads
// are formed: those of the non-basic slacks (B^-1).  An LP of more pivots than
// fit (or with artificials to drive out after phase I) is handed over: its whole
// tableau is formed once and updated at every pivot from there on.
//
// What it saves: a packing LP takes few pivots (8 on average over LPs of 10-500
// rows and columns), and the whole-tableau form writes an FP32 copy of A and
// rewrites it at each of them.  20,000 LPs of those sizes: 10.4 -> 4.9 ms.
#pragma once

#include <climits>

#include "lp_device.cuh"
#include "lp_internal.h"

namespace lpb {
namespace {

__device__ __forceinline__ float fabs32(float v) { return __int_as_float(__float_as_int(v) & INT_MAX); }

// 64-bit key: signed `hi` compared first, then unsigned `lo`.
__device__ __forceinline__ long long pack_key(int hi, unsigned lo) {
    return (long long)(((unsigned long long)(unsigned)hi << 32) | (unsigned long long)lo);
}

struct Tab32 {
    float* T;
    float* colE;
    int* col_var;
    int* row_var;
    int LD;
};

// v <- fma(-b_s, y_s, v), s = max(from, s0) .. to-1 (see chain in
// lp_fp64_deferred.cuh), FP32.
__device__ __forceinline__ float chain32(float v, int s0, int from, int to, const float* bp, int bs, const float* vp,
                                         int vs) {
    bp += (ptrdiff_t)from * bs;
    vp += (ptrdiff_t)from * vs;
#pragma unroll 8
    for (int s = from; s < to; ++s) {
        const float b = -*bp, y = *vp;
        if (s >= s0) v = __fmaf_rn(b, y, v);
        bp += bs;
        vp += vs;
    }
    return v;
}

// One LP's deferred FP32 tableau; all methods are called by every thread of
// the group.  Threads own the rows and the columns congruent to their index.
struct Deferred32 {
    // in `big`
    float *beta, *rf, *obj, *aux;      // right-hand side; the certificate's residual; objective rows
    int *row_last, *negidx, *col_var, *col_last;
    float *cs, *rs;                    // pending pivots [0, ks)
    // in the slot
    float *T, *cg, *rg, *slack;        // whole tableau; pending pivots from ks on; B^-1 columns
    const double* A;
    const int* neg;
    int m, n, W, LD, ks, first, t;
    bool handed;                       // the whole tableau is in T, updated at every pivot
    // pivot t-1's part of the rows' state, applied behind the next barrier
    int rhs_row, rhs_entering;

    __device__ void place(unsigned char* big, size_t big_bytes, unsigned char* slot, int m_, int n_, int k) {
        m = m_;
        n = n_;
        W = n + k + 1;
        const MixedDeferredLayout L = mixed_deferred_layout(m, n, k);
        const MixedDeferredSlot S = mixed_deferred_slot(m, n, k);
        beta = reinterpret_cast<float*>(big + L.beta);
        rf = reinterpret_cast<float*>(big + L.rf);
        row_last = reinterpret_cast<int*>(big + L.row_last);
        negidx = reinterpret_cast<int*>(big + L.negidx);
        obj = reinterpret_cast<float*>(big + L.obj);
        aux = reinterpret_cast<float*>(big + L.aux);
        col_var = reinterpret_cast<int*>(big + L.col_var);
        col_last = reinterpret_cast<int*>(big + L.col_last);
        first = S.first;
        ks = big_bytes > L.hist ? (int)min((size_t)first, (big_bytes - L.hist) / ((size_t)(m + W) * 4)) : 0;
        cs = reinterpret_cast<float*>(big + L.hist);
        rs = cs + (size_t)ks * m;
        T = reinterpret_cast<float*>(slot + S.T);
        LD = S.LD;
        cg = reinterpret_cast<float*>(slot + S.hist) - (ptrdiff_t)ks * m;
        rg = reinterpret_cast<float*>(slot + S.hist) + (size_t)first * m - (ptrdiff_t)ks * W;
        slack = reinterpret_cast<float*>(slot + S.slack);
        t = 0;
        handed = false;
        rhs_row = -1;
    }

    __device__ float* c_at(int s) const { return s < ks ? cs + (size_t)s * m : cg + (ptrdiff_t)s * m; }
    __device__ float* r_at(int s) const { return s < ks ? rs + (size_t)s * W : rg + (ptrdiff_t)s * W; }
    __device__ float ray(int i) const { return c_at(t)[i]; }  // the column formed last

    __device__ float source(int i, int j) const {  // j >= 1
        const float v = (j <= n) ? __double2float_rn(A[(size_t)i * n + j - 1]) : ((neg[j - 1 - n] == i) ? 1.0f : 0.0f);
        return negidx[i] >= 0 ? -v : v;
    }
    // element (i, j) after every pending pivot
    __device__ float element(int i, int j, int sr, int sc) const {
        const int last = max(sr, sc);
        float v;
        if (last < 0) {
            v = source(i, j);
        } else {
            v = r_at(last)[j];
            if (sr < sc) v = __fmaf_rn(-c_at(last)[i], v, 0.0f);
        }
        v = chain32(v, last + 1, last + 1, min(t, ks), cs + i, m, rs + j, W);
        if (t > ks) v = chain32(v, last + 1, max(last + 1, ks), t, cg + i, m, rg + j, W);
        return v;
    }

    // right-hand side, objective rows and labels at the start (row_var and neg
    // are complete)
    template <class G>
    __device__ void build(G& g, const int* row_var, const int* neg_, const double* A_, const double* bv,
                          const double* cv, int k) {
        A = A_;
        neg = neg_;
        const int nm = n + m;
        for (int i = g.tid; i < m; i += g.nt) {
            const bool isneg = row_var[i] >= nm;
            const float v = __double2float_rn(bv[i]);
            beta[i] = isneg ? -v : v;
            negidx[i] = isneg ? row_var[i] - nm : -1;
            row_last[i] = -1;
        }
        g.sync();
        for (int j = g.tid; j < W; j += g.nt) {
            col_last[j] = -1;
            obj[j] = (j >= 1 && j <= n) ? -__double2float_rn(cv[j - 1]) : 0.0f;
            float w = 0.0f;
            for (int u = 0; u < k; ++u) w = __fsub_rn(w, j == 0 ? beta[neg[u]] : source(neg[u], j));
            if (k > 0) aux[j] = w;
        }
    }

    // pivot t-1's right-hand side and row labels (behind a barrier that follows it)
    template <class G>
    __device__ void settle(G& g, int* row_var) {
        if (rhs_row < 0) return;
        const float q0 = r_at(t - 1)[0];
        const float* c = c_at(t - 1);
        for (int i = g.tid; i < m; i += g.nt) {
            if (i == rhs_row) {
                beta[i] = q0;
                row_var[i] = rhs_entering;
                row_last[i] = t - 1;
            } else {
                beta[i] = __fmaf_rn(-c[i], q0, beta[i]);
            }
        }
        rhs_row = -1;
    }
    // column e into c_at(t), each(i, value) for every own row
    template <class G, class F>
    __device__ void column(G& g, int e, F each) {
        const int sc = col_last[e];
        float* dst = c_at(t);
        for (int i = g.tid; i < m; i += g.nt) {
            const float v = element(i, e, row_last[i], sc);
            dst[i] = v;
            each(i, v);
        }
    }
    // The whole tableau after every pending pivot into T, in the whole-tableau
    // form's layout (retired columns 0: their labels keep them out): an LP of
    // many pivots goes on there.  A warp takes 64 columns and kRows rows at a
    // time, with kPivots pivots' entries of the columns in registers and those
    // of the rows one per lane, so that a step waits for one round of loads per
    // 8 x 4 x 64 FMAs.  Bound by that latency: in the tail of a batch an LP's CTA is
    // alone on its SM.  One row at a time against this (packing LPs of A in [1, 10], 48
    // pending pivots, one LP in a hundred handed over): 250 of 150 x 150 0.60 -> 0.50
    // ms, 2500 of 300 x 300 11.1 -> 9.5.
    template <class G>
    __device__ void hand_over(G& g) {
        constexpr int kCols = 2, kPivots = 8, kRows = 4;
        static_assert(kPivots * kRows == 32, "one lane per row and pivot");
        g.sync();  // row_last and col_last as settled
        const int nm = n + m;
        const int strips = (W + 32 * kCols - 1) / (32 * kCols);
        const int groups = max(1, g.nw / strips);  // warps that share a strip of columns, by rows
        for (int w = g.warp; w < strips * groups; w += g.nw) {
            const int strip = w % strips, part = w / strips;
            int j[kCols], sc[kCols];
            bool in[kCols], on[kCols];
#pragma unroll
            for (int q = 0; q < kCols; ++q) {
                j[q] = (strip * kCols + q) * 32 + g.lane;
                in[q] = j[q] >= 1 && j[q] < W;
                if (!in[q]) j[q] = 0;
                on[q] = in[q] && col_var[j[q]] < nm;
                sc[q] = on[q] ? col_last[j[q]] : t;  // t: no step applies
            }
            for (int p0 = 0; p0 == 0 || p0 < t; p0 += kPivots) {
                float r[kPivots][kCols];
#pragma unroll
                for (int u = 0; u < kPivots; ++u)
#pragma unroll
                    for (int q = 0; q < kCols; ++q) r[u][q] = on[q] && p0 + u < t ? r_at(p0 + u)[j[q]] : 0.0f;
                for (int i0 = part * kRows; i0 < m; i0 += groups * kRows) {
                    const int ls = p0 + g.lane / kRows, li = i0 + g.lane % kRows;
                    const float c = ls < t && li < m ? -c_at(ls)[li] : 0.0f;
                    int sr[kRows];
                    float v[kRows][kCols];
#pragma unroll
                    for (int a = 0; a < kRows; ++a) {
                        const int i = min(i0 + a, m - 1);  // past the last row: that row again, not stored
                        sr[a] = row_last[i];
#pragma unroll
                        for (int q = 0; q < kCols; ++q) {
                            v[a][q] = 0.0f;
                            if (p0 > 0 && on[q]) v[a][q] = T[(size_t)i * LD + j[q]];
                            else if (on[q] && sr[a] < 0 && sc[q] < 0) v[a][q] = source(i, j[q]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kPivots; ++u) {
                        const int s = p0 + u;
                        if (s < t) {
#pragma unroll
                            for (int a = 0; a < kRows; ++a) {
                                const float b = __shfl_sync(kFull, c, u * kRows + a);
#pragma unroll
                                for (int q = 0; q < kCols; ++q) {
                                    const int last = max(sr[a], sc[q]);
                                    if (s == last) v[a][q] = (sr[a] >= sc[q]) ? r[u][q] : __fmaf_rn(b, r[u][q], 0.0f);
                                    else if (s > last) v[a][q] = __fmaf_rn(b, r[u][q], v[a][q]);
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int a = 0; a < kRows; ++a)
#pragma unroll
                        for (int q = 0; q < kCols; ++q)
                            if (in[q] && i0 + a < m) T[(size_t)(i0 + a) * LD + j[q]] = v[a][q];
                }
            }
        }
        for (int i = g.tid; i < m; i += g.nt) T[(size_t)i * LD] = beta[i];
        for (int j = g.tid; j < W; j += g.nt) {
            T[(size_t)m * LD + j] = obj[j];
            T[(size_t)(m + 1) * LD + j] = aux[j];
        }
        handed = true;
        g.sync();
    }
    // Step 3's row for column j: r_t and the objective row(s) (`both`: phase I's two)
    __device__ void scale(int j, float u, int e, float rinv, float de, float dw, bool both) {
        const float p = (j == e) ? rinv : __fmul_rn(u, rinv);
        r_at(t)[j] = p;
        obj[j] = __fmaf_rn(-de, p, (j == e) ? 0.0f : obj[j]);
        if (both) aux[j] = __fmaf_rn(-dw, p, (j == e) ? 0.0f : aux[j]);
    }

    // Steps 1-3 until the LP halts (Section 3, two-phase method), with the
    // whole-tableau form's decisions.
    template <class G>
    __device__ void simplex(G& g, Tab32& tb, const Tolerances& tol, const MixedParams& mp, int32_t* diag, int lp,
                            double bmax, int max_iters, int& status, int& phase, int& iters, int& e_unb) {
        const int tid = g.tid, nt = g.nt, nm = n + m;
        int* row_var = tb.row_var;
        const int key_neg_eps_opt = fkey(-mp.eps_opt32);
        while (status < 0) {
            const bool one = phase == 1;
            const float* orow = one ? aux : obj;
            bool end_phase1 = false;
            // Step 1 (own columns: written by this thread)
            long long dloc = LLONG_MAX;
            for (int j = tid; j < W; j += nt) {
                const int v = col_var[j];
                if (j >= 1 && v < nm) dloc = min(dloc, pack_key(fkey(orow[j]), ((unsigned)v << 16) | (unsigned)j));
            }
            const long long dsel = g.min_i64(dloc);
            settle(g, row_var);
            const int dmin = (int)(dsel >> 32);
            if (dsel == LLONG_MAX || dmin >= key_neg_eps_opt) {
                if (!one) { status = kOptimal; break; }
                end_phase1 = true;
            } else {
                const int e = (int)(dsel & 0xffff);
                if (e < 1 || e >= W) {
                    if (tid == 0) record_internal_error(diag, 1, lp, dmin, 0, iters, phase, (int)(dsel & 0xffffffff));
                    status = kNumerical;
                    break;
                }
                if (t == first) {
                    hand_over(g);
                    return;
                }
                // Step 2
                const float de = obj[e], dw = one ? aux[e] : 0.0f;
                long long rloc = LLONG_MAX;
                column(g, e, [&](int i, float te) {
                    if (te > mp.eps_piv32) rloc = min(rloc, pack_key(fkey(__fdividef(beta[i], te)), (unsigned)i));
                });
                const long long rsel = g.min_i64(rloc);
                if (rsel == LLONG_MAX) {
                    if (!one) {
                        status = kUnbounded;
                        e_unb = e;
                        break;
                    }
                    end_phase1 = true;  // FP32 noise in the auxiliary row (the certificate decides)
                } else {
                    const int l = (int)(rsel & 0xffffffff);
                    if (l < 0 || l >= m) {
                        if (tid == 0) record_internal_error(diag, 2, lp, (int)(rsel >> 32), 0, iters, phase, l);
                        status = kNumerical;
                        break;
                    }
                    const float pe = c_at(t)[l];
                    if (!isfinite(pe)) { status = kNumerical; break; }
                    if (iters >= max_iters) { status = kIterLimit; break; }
                    // Step 3
                    const float rinv = __frcp_rn(pe);
                    const int left = row_var[l], sr = row_last[l];  // rewritten behind the next barrier (settle)
                    for (int j = tid; j < W; j += nt) {
                        if (j == 0) scale(0, beta[l], e, rinv, de, dw, one);
                        else if (col_var[j] < nm) scale(j, element(l, j, sr, col_last[j]), e, rinv, de, dw, one);
                    }
                    finish(tid, nt, e, l, (int)((dsel >> 16) & 0xffff), left);
                    ++iters;
                }
            }
            if (end_phase1) {
                g.sync();  // row labels as settled
                if (-aux[0] > mp.eps_feas32 * (float)bmax) { status = kInfeasible; break; }
                unsigned basic = 0xffffffffu;  // an artificial still basic, to be driven out
                for (int i = tid; i < m; i += nt)
                    if (row_var[i] >= nm) basic = 0;
                if (g.min_u32(basic) == 0u) {
                    hand_over(g);
                    return;
                }
                phase = 2;
            }
        }
        g.sync();
        settle(g, row_var);
        g.sync();
    }
    // labels of pivot t on (l, e): the column's by its owner now, the row's in settle
    __device__ void finish(int tid, int nt, int e, int l, int entering, int left) {
        if (tid == e % nt) {
            col_var[e] = left;  // an artificial (>= n + m) retires with its column
            col_last[e] = t;
        }
        rhs_row = l;
        rhs_entering = entering;
        ++t;
    }

    // The columns of the non-basic slacks nbl[0 .. nnb) (position << 16 | slack),
    // one after the other, for the certificate.
    template <class G>
    __device__ void slack_columns(G& g, const int* nbl, int nnb) {
        for (int u = 0; u < nnb; ++u) {
            const int j = (int)((unsigned)nbl[u] >> 16), sc = col_last[j];
            for (int i = g.tid; i < m; i += g.nt) slack[(size_t)u * m + i] = element(i, j, row_last[i], sc);
        }
        g.sync();
    }
};

}  // namespace
}  // namespace lpb
