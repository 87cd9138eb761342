// lp_prepare.cu -- input checks, per-LP phase-I row counts and signs, run once by
// lp_batch_create to plan the launches (the batch sizing of Algorithm 1 in
// Section 4.1 needs each LP's tableau footprint, Eq. 5).  The check runs on
// the batch's own copy of the inputs and zeroes every non-finite entry it
// counts, so that no kernel after it on the stream sees one, whether or not
// the host has read the count yet.

#include <climits>

#include "lp_internal.h"

namespace lpb {
namespace {

// Counts the non-finite entries of v into *bad and sets them to 0.
__global__ void check_finite_kernel(double* __restrict__ v, int64_t len, unsigned long long* bad) {
    unsigned long long local = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
        const long long bits = __double_as_longlong(v[i]) & LLONG_MAX;
        if (bits >= 0x7FF0000000000000LL) {
            v[i] = 0.0;
            ++local;
        }
    }
    local = __reduce_add_sync(0xffffffffu, (unsigned)local);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(bad, local);
}

// One warp per LP: number of rows with b_i < 0 (rows that get an artificial),
// with kPlanSigned added unless A was seen to have no negative entry, and
// kPlanSameA when A is the previous LP's (its sign is then not looked for).  A
// sample of A is read (SignLook), and only where its sign matters to the plan: a
// wrong guess costs time, not results.
__global__ void plan_info_kernel(const DeviceBatch B, int32_t num_lps, SignLook look, int32_t* __restrict__ info) {
    const int lane = threadIdx.x & 31;
    const int lp = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (lp >= num_lps) return;
    const int m = B.m[lp], n = B.n[lp];
    const double* bv = B.b + B.b_off[lp];
    int cnt = 0;
    for (int i = lane; i < m; i += 32) cnt += (bv[i] < 0.0) ? 1 : 0;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    int flags = kPlanSigned;  // where it was not looked for
    if (look != kLookNot && sign_matters(m, n)) {
        if (lp > 0 && B.a_off[lp] == B.a_off[lp - 1] && m == B.m[lp - 1] && n == B.n[lp - 1]) {
            flags = kPlanSameA;
        } else {
            flags = 0;
            const double* A = B.A + B.a_off[lp];
            const int64_t len = (int64_t)m * n;
            for (int i = 0; i < sign_samples(look) && !flags; i += 256) {
                bool negative = false;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int64_t at = sign_sample_at(look, len, i + q * 32 + lane);
                    negative |= at < len && A[at] < 0.0;
                }
                if (__any_sync(0xffffffffu, negative)) flags = kPlanSigned;
            }
        }
    }
    if (lane == 0) info[lp] = cnt | flags;
}

// Array blockIdx.y of the list, in 16-byte pieces where both ends allow it.
// Bound by the launch for small batches (five separate copies were most of a
// 5 x 5 batch's results), by HBM for large ones.
__global__ void __launch_bounds__(256) copy_list_kernel(const __grid_constant__ CopyList list) {
    const int a = blockIdx.y;
    const size_t stride = (size_t)gridDim.x * blockDim.x, t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t bytes = list.bytes[a];
    size_t done = 0;
    if (((reinterpret_cast<uintptr_t>(list.dst[a]) | reinterpret_cast<uintptr_t>(list.src[a])) & 15u) == 0) {
        const uint4* src = static_cast<const uint4*>(list.src[a]);
        uint4* dst = static_cast<uint4*>(list.dst[a]);
        const size_t n = bytes / 16;
#pragma unroll 4
        for (size_t i = t0; i < n; i += stride) dst[i] = src[i];
        done = n * 4;
    }
    const uint32_t* src = static_cast<const uint32_t*>(list.src[a]);
    uint32_t* dst = static_cast<uint32_t*>(list.dst[a]);
    for (size_t i = done + t0; i < bytes / 4; i += stride) dst[i] = src[i];
}

int grid_for(int64_t len, int threads) {
    int64_t g = (len + threads * 4 - 1) / (threads * 4);
    if (g < 1) g = 1;
    if (g > 4096) g = 4096;
    return (int)g;
}

}  // namespace

cudaError_t launch_input_check(double* A, int64_t a_len, double* b, int64_t b_len, double* c, int64_t c_len,
                               unsigned long long* bad, cudaStream_t stream) {
    cudaError_t err = cudaMemsetAsync(bad, 0, sizeof(unsigned long long), stream);
    if (err != cudaSuccess) return err;
    const int t = 256;
    if (a_len > 0) check_finite_kernel<<<grid_for(a_len, t), t, 0, stream>>>(A, a_len, bad);
    if (b_len > 0) check_finite_kernel<<<grid_for(b_len, t), t, 0, stream>>>(b, b_len, bad);
    if (c_len > 0) check_finite_kernel<<<grid_for(c_len, t), t, 0, stream>>>(c, c_len, bad);
    return cudaGetLastError();
}

cudaError_t launch_plan_info(const DeviceBatch& B, int32_t num_lps, SignLook look, int32_t* info,
                             cudaStream_t stream) {
    const int t = 256;
    const int64_t threads = (int64_t)num_lps * 32;
    plan_info_kernel<<<(unsigned)((threads + t - 1) / t), t, 0, stream>>>(B, num_lps, look, info);
    return cudaGetLastError();
}

cudaError_t launch_copy_list(const CopyList& list, cudaStream_t stream) {
    size_t most = 0;
    for (int i = 0; i < list.count; ++i) most = list.bytes[i] > most ? list.bytes[i] : most;
    // four 16-byte pieces per thread, at most 8 CTAs per SM (of 152) for each array
    const size_t blocks = (most + 16383) / 16384;
    copy_list_kernel<<<dim3((unsigned)(blocks < 1 ? 1 : (blocks > 1216 ? 1216 : blocks)), list.count), 256, 0, stream>>>(
        list);
    return cudaGetLastError();
}

}  // namespace lpb
