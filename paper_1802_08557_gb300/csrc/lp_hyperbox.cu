// lp_hyperbox.cu -- hyperbox LPs (Gurung & Ray, arXiv 1802.08557, Section
// 4.4, Eq. 7): maximise l.x over a box lo <= x <= hi for many directions l.
// The maximiser takes lo_i where l_i < 0 and hi_i otherwise, so each LP is one
// dot product sum_i l_i h_i.
//
// The paper gives each LP a 32-thread block with one working thread.  Here:
//  - dim <= kTileMaxDim: persistent CTAs stride over tiles of `tile_lps`
//    consecutive LPs; each tile (l, and the per-LP boxes when there are any)
//    is staged into shared memory by bulk asynchronous copies (cp.async.bulk,
//    completion counted on an mbarrier), `stages` tiles in flight per CTA.
//    Thread t then owns LP t of the tile: obj = fma over i = 0..dim-1 in index
//    order, h_i chosen by a 32-bit integer sign test (no FP64 compare), the shared
//    box read from shared memory (a broadcast).  A thread reads 4 coordinates per
//    step in 16-byte loads where dim allows it (2, or 1): with 8-byte loads the
//    rows of a warp, 8 dim bytes apart, met in the same banks for an even dim
//    (16-way for 16, 32, 48, 64).  2^22 LPs, one box, us, 8-byte loads and tiles of
//    128 before: dim 16 277 -> 123, dim 28 241 -> 209, dim 32 531 -> 247; 2^21 of
//    dim 64 689 -> 315.  x, when asked for, is written
//    by a flat pass over the tile (coalesced stores).  Tiles that are not
//    whole (the last one) or arrays that are not 16-byte aligned are loaded
//    with plain loads instead.
//  - larger dim: a warp's lanes over i, a fixed xor-tree sum, up to 8 LPs per warp.
// Bound: the FP64 pipe (one FMA per 8 bytes of l) for one shared box and no x;
// HBM bandwidth when every LP has its own box or x is written.
//
// Waits on an mbarrier are bounded (kWaitCycles of clock64): a CTA whose copy
// does not complete gives up, writes NaN to the outputs of the tiles it has
// not finished, waits (bounded again) for its other copies and returns.

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "lp_internal.h"

namespace lpb {
namespace {

constexpr int kTileMaxDim = 64;
constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz
constexpr unsigned kFullMask = 0xffffffffu;

struct HbArgs {
    const double* L;
    const double* lo;
    const double* hi;
    double* obj;
    double* x;
    int64_t num_lps;
    int64_t num_tiles;
    int64_t num_full_tiles;  // tiles that may be bulk-copied (whole, aligned)
    int dim;
    int tile_lps;            // LPs per tile = threads per CTA
    int stages;
    int stage_offset;        // bytes from the start of shared memory
    int stage_bytes;
};

// l < 0 (strictly: -0 is not negative), from the bits, in 32-bit words: on
// GB300 a 64-bit integer compare, like an FP64 compare, is issued to the
// FP64 pipe, where it would cost as much as the FMA it feeds (measured: one
// such test per coordinate halved the kernel's FMA rate).
__device__ __forceinline__ bool is_negative(double v) {
    const unsigned hw = (unsigned)__double2hiint(v);
    const unsigned lw = (unsigned)__double2loint(v);
    return (hw >> 31) != 0u && ((hw << 1) | lw) != 0u;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// Bulk copy global -> this CTA's shared memory; bytes a multiple of 16, both
// addresses 16-byte aligned.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Order this thread's earlier generic-proxy accesses of shared memory before
// later async-proxy (bulk copy) writes to it.
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Wait for the phase with the given parity; false after kWaitCycles.
__device__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > kWaitCycles) return false;
    return true;
}

// The bit of the lane that tells apart the lanes of a quarter warp whose rows
// (8 dim bytes apart, dim a multiple of 4) start in the same bank.
__device__ __forceinline__ int swap_shift(int dim) { return dim % 16 == 0 ? 0 : (dim % 8 == 0 ? 1 : 2); }

// kWidth: coordinates per step, a divisor of dim (1, 2 or 4).
template <bool kBoxPerLp, int kWidth>
__global__ void __launch_bounds__(128) hyperbox_tile_kernel(const HbArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);        // one per stage
    double* box = reinterpret_cast<double*>(smem + 64);       // shared box: lo, hi
    const int tid = threadIdx.x, nt = blockDim.x;
    const int dim = a.dim;
    const int S = a.stages;
    const int64_t tile_elems = (int64_t)a.tile_lps * dim;
    const uint32_t tile_bytes = (uint32_t)(tile_elems * 8);

    if (tid == 0) {
        for (int s = 0; s < S; ++s) mbar_init(&bar[s], 1);
        mbar_init_fence();
    }
    if (!kBoxPerLp)
        for (int i = tid; i < dim; i += nt) {
            box[i] = a.lo[i];
            box[dim + i] = a.hi[i];
        }
    __syncthreads();

    auto stage = [&](int s) { return reinterpret_cast<double*>(smem + a.stage_offset + (size_t)s * a.stage_bytes); };
    auto issue = [&](int64_t t, int s) {  // thread 0 only
        double* d = stage(s);
        const int64_t off = t * tile_elems;
        mbar_expect_tx(&bar[s], kBoxPerLp ? 3u * tile_bytes : tile_bytes);
        bulk_load(d, a.L + off, tile_bytes, &bar[s]);
        if (kBoxPerLp) {
            bulk_load(d + tile_elems, a.lo + off, tile_bytes, &bar[s]);
            bulk_load(d + 2 * tile_elems, a.hi + off, tile_bytes, &bar[s]);
        }
    };

    const int64_t t0 = blockIdx.x, step = gridDim.x;
    uint32_t pending = 0;  // stages with a copy issued and not yet waited for (thread 0's view)
    if (tid == 0)
        for (int s = 0; s < S; ++s) {
            const int64_t t = t0 + (int64_t)s * step;
            if (t < a.num_full_tiles) {
                issue(t, s);
                pending |= 1u << s;
            }
        }
    uint32_t phase = 0;  // bit s: parity of the next completion of stage s
    bool ok = true;
    for (int64_t it = 0;; ++it) {
        const int64_t t = t0 + it * step;
        if (t >= a.num_tiles) break;
        const int s = (int)(it % S);
        double* Ls = stage(s);
        const int64_t lp0 = t * a.tile_lps;
        const int count = (int)((a.num_lps - lp0) < a.tile_lps ? (a.num_lps - lp0) : a.tile_lps);
        const int64_t n_el = (int64_t)count * dim;
        if (t < a.num_full_tiles) {
            bool got = ok && mbar_wait(&bar[s], (phase >> s) & 1u);
            got = __syncthreads_and(got) != 0;
            if (got) {
                phase ^= 1u << s;
                pending &= ~(1u << s);
            }
            ok = got;
        } else if (ok) {
            // plain loads: the last (partial) tile, or arrays that are not aligned
            const int64_t g0 = lp0 * dim;
            for (int64_t e = tid; e < n_el; e += nt) {
                Ls[e] = a.L[g0 + e];
                if (kBoxPerLp) {
                    Ls[tile_elems + e] = a.lo[g0 + e];
                    Ls[2 * tile_elems + e] = a.hi[g0 + e];
                }
            }
            __syncthreads();
        }
        if (!ok) {
            // a copy did not complete: no result for this tile
            const double nan = __longlong_as_double(0x7FF8000000000000LL);
            if (tid < count) a.obj[lp0 + tid] = nan;
            if (a.x)
                for (int64_t e = tid; e < n_el; e += nt) a.x[lp0 * dim + e] = nan;
            continue;
        }
        if (tid < count) {
            const double* l = Ls + (size_t)tid * dim;
            const double* lo = kBoxPerLp ? Ls + tile_elems + (size_t)tid * dim : box;
            const double* hi = kBoxPerLp ? Ls + 2 * tile_elems + (size_t)tid * dim : box + dim;
            double acc = 0.0;
            auto step = [&](double li, double lv, double hv) { acc = __fma_rn(li, is_negative(li) ? lv : hv, acc); };
            if (kWidth == 4) {
                // lanes that would meet in a bank read the two halves of their four
                // coordinates in opposite order
                const int first = ((tid >> swap_shift(dim)) & 1) * 2, second = 2 - first;
                for (int i = 0; i < dim; i += 4) {
                    const double2 p = *reinterpret_cast<const double2*>(l + i + first);
                    const double2 q = *reinterpret_cast<const double2*>(l + i + second);
                    double2 lo0, lo1, hi0, hi1;
                    if (kBoxPerLp) {
                        const double2 a0 = *reinterpret_cast<const double2*>(lo + i + first);
                        const double2 a1 = *reinterpret_cast<const double2*>(lo + i + second);
                        const double2 b0 = *reinterpret_cast<const double2*>(hi + i + first);
                        const double2 b1 = *reinterpret_cast<const double2*>(hi + i + second);
                        lo0 = first ? a1 : a0, lo1 = first ? a0 : a1;
                        hi0 = first ? b1 : b0, hi1 = first ? b0 : b1;
                    } else {
                        lo0 = *reinterpret_cast<const double2*>(lo + i), lo1 = *reinterpret_cast<const double2*>(lo + i + 2);
                        hi0 = *reinterpret_cast<const double2*>(hi + i), hi1 = *reinterpret_cast<const double2*>(hi + i + 2);
                    }
                    const double2 l0 = first ? q : p, l1 = first ? p : q;
                    step(l0.x, lo0.x, hi0.x);
                    step(l0.y, lo0.y, hi0.y);
                    step(l1.x, lo1.x, hi1.x);
                    step(l1.y, lo1.y, hi1.y);
                }
            } else if (kWidth == 2) {
#pragma unroll 2
                for (int i = 0; i < dim; i += 2) {
                    const double2 l2 = *reinterpret_cast<const double2*>(l + i);
                    const double2 lo2 = *reinterpret_cast<const double2*>(lo + i);
                    const double2 hi2 = *reinterpret_cast<const double2*>(hi + i);
                    step(l2.x, lo2.x, hi2.x);
                    step(l2.y, lo2.y, hi2.y);
                }
            } else {
#pragma unroll 4
                for (int i = 0; i < dim; ++i) {
                    const double li = l[i];
                    acc = __fma_rn(li, is_negative(li) ? lo[i] : hi[i], acc);
                }
            }
            a.obj[lp0 + tid] = acc;
        }
        if (a.x) {
            // h, coalesced: element e of the tile is coordinate e mod dim
            const int dstep = nt % dim;
            int i = tid % dim;
            for (int64_t e = tid; e < n_el; e += nt) {
                const double li = Ls[e];
                double h;
                if (kBoxPerLp) h = is_negative(li) ? Ls[tile_elems + e] : Ls[2 * tile_elems + e];
                else h = is_negative(li) ? box[i] : box[dim + i];
                a.x[lp0 * dim + e] = h;
                i += dstep;
                if (i >= dim) i -= dim;
            }
        }
        __syncthreads();  // every thread is done with stage s
        if (tid == 0) {
            const int64_t tn = t + (int64_t)S * step;
            if (tn < a.num_full_tiles) {
                fence_proxy_async();
                issue(tn, s);
                pending |= 1u << s;
            }
        }
    }
    // after a failed wait: let the copies still in flight land before exiting
    if (tid == 0 && !ok)
        for (int s = 0; s < S; ++s)
            if (pending & (1u << s)) mbar_wait(&bar[s], (phase >> s) & 1u);
}

// kLps LPs per warp.  The xor-tree sum of one LP by itself is 5 adds of the whole
// warp, as much FP64 pipe as 160 coordinates; for 8 LPs together each step halves
// the LPs that a lane still carries: 4 + 2 + 1 + 1 + 1 adds, the same sums; and 8
// rows' loads are in flight.  One LP per warp against 8, one box, us: 400,000 of
// dim 65 231 -> 112, of dim 160 311 -> 161; 4 LPs and a box each, 150,000 of dim
// 100: 103 -> 71.  80 registers, three CTAs per SM (64 spill).
template <bool kBoxPerLp, int kLps>
__global__ void __launch_bounds__(256, 3) hyperbox_warp_kernel(const HbArgs a) {
    const int lane = threadIdx.x & 31;
    const int dim = a.dim;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k = w0 * kLps; k < a.num_lps; k += nw * kLps) {
        const int last = (int)(a.num_lps - 1 - k < kLps - 1 ? a.num_lps - 1 - k : kLps - 1);
        const int64_t base = k * dim;
        double acc[kLps];
#pragma unroll
        for (int q = 0; q < kLps; ++q) acc[q] = 0.0;
        const double *L = a.L + base + lane, *lo = a.lo + lane, *hi = a.hi + lane;
        if (kBoxPerLp) lo += base, hi += base;
        double* x = a.x ? a.x + base + lane : nullptr;
#pragma unroll 1
        for (int i = lane; i < dim; i += 32, L += 32, lo += 32, hi += 32) {
            double li[kLps], l0[kLps], h0[kLps];
            int at = 0;
#pragma unroll
            for (int q = 0; q < kLps; ++q) {
                li[q] = L[at];
                l0[q] = (kBoxPerLp || q == 0) ? lo[at] : l0[0];
                h0[q] = (kBoxPerLp || q == 0) ? hi[at] : h0[0];
                if (q < last) at += dim;  // past the last LP: its row again, not stored
            }
            at = 0;
#pragma unroll
            for (int q = 0; q < kLps; ++q) {
                l0[q] = is_negative(li[q]) ? l0[q] : h0[q];
                acc[q] = __fma_rn(li[q], l0[q], acc[q]);
            }
            if (x) {
#pragma unroll
                for (int q = 0; q < kLps; ++q, at += dim)
                    if (q <= last) x[at] = l0[q];
                x += 32;
            }
        }
        int o = 16, lp = 0;
#pragma unroll
        for (int w = kLps / 2; w > 0; w >>= 1, o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int q = 0; q < w; ++q) {
                const double keep = up ? acc[q + w] : acc[q], give = up ? acc[q] : acc[q + w];
                acc[q] = __dadd_rn(keep, __shfl_xor_sync(kFullMask, give, o));
            }
            if (up) lp += w;
        }
#pragma unroll
        for (; o > 0; o >>= 1) acc[0] = __dadd_rn(acc[0], __shfl_xor_sync(kFullMask, acc[0], o));
        if ((lane & (32 / kLps - 1)) == 0 && lp <= last) a.obj[k + lp] = acc[0];
    }
}

int g_num_sms[64] = {};

int num_sms(int device) {
    if (device < 0 || device >= 64) return 152;
    if (g_num_sms[device] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || v <= 0) v = 152;
        g_num_sms[device] = v;
    }
    return g_num_sms[device];
}

}  // namespace

cudaError_t launch_hyperbox(const double* L, const double* lo, const double* hi, bool box_per_lp, double* obj,
                            double* x, int64_t num_lps, int dim, cudaStream_t stream) {
    if (num_lps <= 0) return cudaSuccess;
    int device = 0;
    cudaError_t err = cudaGetDevice(&device);
    if (err != cudaSuccess) return err;
    const int sms = num_sms(device);
    HbArgs a{};
    a.L = L; a.lo = lo; a.hi = hi; a.obj = obj; a.x = x;
    a.num_lps = num_lps;
    a.dim = dim;
    if (dim > kTileMaxDim) {
        // 8 LPs per warp (4 with a box each: registers) from 16 warps per SM on; below
        // that one each, for latency (10,000 of dim 100: 10 us either way)
        const int per_warp = num_lps >= (int64_t)sms * 128 ? (box_per_lp ? 4 : 8) : 1;
        const int threads = 256;
        const int64_t blocks = std::min<int64_t>((num_lps + 8 * per_warp - 1) / (8 * per_warp), (int64_t)sms * 8);
        auto kernel = per_warp > 1 ? (box_per_lp ? hyperbox_warp_kernel<true, 4> : hyperbox_warp_kernel<false, 8>)
                                   : (box_per_lp ? hyperbox_warp_kernel<true, 1> : hyperbox_warp_kernel<false, 1>);
        kernel<<<(unsigned)blocks, threads, 0, stream>>>(a);
        return cudaGetLastError();
    }
    const int arrays = box_per_lp ? 3 : 1;
    // Rows of more than 12 doubles (8 with a box each): one warp per CTA and two
    // stages, as many CTAs as fit, so that the FP64 pipe and the copies of an SM
    // never wait for one CTA's barrier.  2^22 LPs of dim 28, one box: 209 us against
    // 211, 217 and 235 with tiles of 64, 96 and 128, 219 with three stages; 2^20 with
    // a box and x each 164, 193 (64 and 128), 252 (three stages).  Short rows: tiles
    // of 128, where a tile's fixed cost counts (dim 2: 27 us against 31 with tiles of
    // 32; dim 5 with boxes and x, 2 M LPs: 54 against 56), and up to 40 KB in flight
    // per CTA (dim 12: 95 us with three stages, 99 with four, 100 with two).
    const bool short_rows = dim <= (box_per_lp ? 8 : 12);
    a.tile_lps = short_rows ? 128 : 32;
    a.stage_bytes = (int)((size_t)a.tile_lps * dim * 8 * arrays);
    a.stages = short_rows ? std::max(2, std::min(4, (40 << 10) / a.stage_bytes)) : 2;
    a.stage_offset = ((64 + 2 * dim * 8 + 127) / 128) * 128;  // mbarriers, shared box, then the stages
    const size_t smem = (size_t)a.stage_offset + (size_t)a.stages * a.stage_bytes;
    a.num_tiles = (num_lps + a.tile_lps - 1) / a.tile_lps;
    auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    const bool bulk = aligned(L) && (!box_per_lp || (aligned(lo) && aligned(hi)));
    a.num_full_tiles = bulk ? num_lps / a.tile_lps : 0;
    auto kernel = dim % 4 == 0   ? (box_per_lp ? hyperbox_tile_kernel<true, 4> : hyperbox_tile_kernel<false, 4>)
                  : dim % 2 == 0 ? (box_per_lp ? hyperbox_tile_kernel<true, 2> : hyperbox_tile_kernel<false, 2>)
                                 : (box_per_lp ? hyperbox_tile_kernel<true, 1> : hyperbox_tile_kernel<false, 1>);
    if ((err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return err;
    int per_sm = 0;
    if ((err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, a.tile_lps, smem))) return err;
    const int64_t blocks = std::min<int64_t>(a.num_tiles, (int64_t)sms * std::max(1, per_sm));
    kernel<<<(unsigned)blocks, a.tile_lps, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace lpb
