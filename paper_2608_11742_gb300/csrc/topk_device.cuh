// topk_device.cuh -- warp-wide top-k lists: lane j holds rank j of a list of
// (logit, token) pairs, logit descending, then token ascending.
#pragma once

#include <climits>

#include "rps_internal.cuh"

namespace rps {
namespace {

constexpr int kCandBatch = 32;  // candidates merged at a time

// True when (av, ai) ranks before (bv, bi): larger logit, then lower token id.
__device__ __forceinline__ bool ranks_before(float av, int ai, float bv, int bi) {
    return av > bv || (av == bv && ai < bi);
}

// The 32 lane values in descending order, lane j holding rank j (bitonic sort).
__device__ __forceinline__ float warp_sort_desc(float x, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const float o = __shfl_xor_sync(kFull, x, stride);
            const bool keep_max = ((lane & size) == 0) == ((lane & stride) == 0);
            x = keep_max ? fmaxf(x, o) : fminf(x, o);
        }
    }
    return x;
}

// k-th largest of the 32 lane values, 1 <= k <= 32.
__device__ __forceinline__ float warp_kth_largest(float x, int k, int lane) {
    return __shfl_sync(kFull, warp_sort_desc(x, lane), k - 1);
}

// k-th largest of 64 values, two per lane, 1 <= k <= 32: with both sets sorted,
// the largest over i of the smaller of the i-th of one and the (k - i)-th of
// the other (each choice takes k values, the best one the k largest).
__device__ __forceinline__ float warp_kth_largest2(float x, float y, int k, int lane) {
    x = warp_sort_desc(x, lane);
    y = warp_sort_desc(y, lane);
    const int j = k - 1 - (lane + 1);  // lane: ranks 0..lane of x with ranks 0..j of y (none when j == -1)
    const float yj = __shfl_sync(kFull, y, max(j, 0));
    const float yk = __shfl_sync(kFull, y, k - 1);
    float v = j >= -1 ? (j >= 0 ? fminf(x, yj) : x) : -INFINITY;
    return fmaxf(warp_max(v), yk);
}

// Merges one candidate per lane (sentinel -inf / INT_MAX for none) into the
// warp-distributed sorted list: bitonic sort of the 32 candidates in rank order,
// then the element-wise better of the list and the reversed candidates (the 32
// best of both, as a bitonic sequence), then a bitonic merge. Fixed cost,
// independent of how many candidates are real.
__device__ __forceinline__ void pair_step(float &v, int &i, int stride, bool keep_better) {
    const float ov = __shfl_xor_sync(kFull, v, stride);
    const int oi = __shfl_xor_sync(kFull, i, stride);
    if (keep_better == ranks_before(ov, oi, v, i)) {
        v = ov;
        i = oi;
    }
}

// The list holds nothing yet: each real candidate's rank among the 32 is the
// count of candidates before it (candidates are distinct, so ranks are); ranks
// below k go to buf[rank] (kCandBatch entries), then lane j takes rank j.
// Independent shuffles instead of a sorting network's dependent stages.
__device__ __forceinline__ void warp_rank_into_list(float &tv, int &ti, float cv, int ci, int k, int lane,
                                                    float2 *buf) {
    const bool real = ci != INT_MAX;
    int rank = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float ov = __shfl_sync(kFull, cv, j);
        const int oi = __shfl_sync(kFull, ci, j);
        rank += ranks_before(ov, oi, cv, ci);
    }
    const int n = __popc(__ballot_sync(kFull, real));
    __syncwarp();
    if (real && rank < k) buf[rank] = make_float2(cv, __int_as_float(ci));
    __syncwarp();
    const float2 e = lane < k && lane < n ? buf[lane] : make_float2(-INFINITY, __int_as_float(INT_MAX));
    tv = e.x;
    ti = __float_as_int(e.y);
    __syncwarp();
}

__device__ __forceinline__ void warp_merge_batch(float &tv, int &ti, float cv, int ci, int k, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1)
            pair_step(cv, ci, stride, ((lane & size) == 0) == ((lane & stride) == 0));
    }
    const float rv = __shfl_sync(kFull, cv, 31 - lane);
    const int ri = __shfl_sync(kFull, ci, 31 - lane);
    if (ranks_before(rv, ri, tv, ti)) {
        tv = rv;
        ti = ri;
    }
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) pair_step(tv, ti, stride, (lane & stride) == 0);
    if (lane >= k) {
        tv = -INFINITY;
        ti = INT_MAX;
    }
}

}  // namespace
}  // namespace rps
