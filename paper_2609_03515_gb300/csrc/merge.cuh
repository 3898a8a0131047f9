// Merge of a head's split-K partials, by one warp.
#pragma once
#include "ikv_internal.cuh"

namespace ikv {
namespace {

__device__ __forceinline__ void store_as(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void store_as(float *p, float v) { *p = v; }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ml: the head's n <= kMaxSplits (max, sum) pairs, po: its partial outputs [n][32 E]; out gets
// their merged output (32 E values), lse2 (or null) the log2-sum-exp.  wq: kMaxSplits floats
// of shared memory of the calling warp.  The (max, sum) pairs give each partial's weight, then
// every lane sums E output dims over the partials, eight loads in flight.
template <int E, typename T>
__device__ __forceinline__ void merge_head(const float2 *ml, const float *po, int n, float *wq, T *out, float *lse2) {
    const int lane = threadIdx.x & 31;
    po += lane * E;
    float mv[kMaxSplits / 32], lv[kMaxSplits / 32], M = -INFINITY;
#pragma unroll
    for (int k = 0; k < kMaxSplits / 32; ++k) {
        const int q = lane + 32 * k;
        const float2 x = q < n ? __ldcg(ml + q) : make_float2(-INFINITY, 0.f);
        mv[k] = x.x;
        lv[k] = x.y;
        M = fmaxf(M, x.x);
    }
    M = warp_max(M);
    const float ref = M == -INFINITY ? 0.f : M;  // every slot dead: nothing to scale
    float W = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxSplits / 32; ++k) {
        const float f = exp2f(mv[k] - ref);
        W += lv[k] * f;
        wq[lane + 32 * k] = f;
    }
    W = warp_sum(W);
    __syncwarp();
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    for (int q0 = 0; q0 < n; q0 += 8) {
        float ov[8][E];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float *p = po + (int64_t)(q0 + j) * 32 * E;
            if (E == 4) {
                const float4 x = q0 + j < n ? __ldcg(reinterpret_cast<const float4 *>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
                ov[j][0] = x.x;
                ov[j][1] = x.y;
                ov[j][E - 2] = x.z;
                ov[j][E - 1] = x.w;
            } else {
                const float2 x = q0 + j < n ? __ldcg(reinterpret_cast<const float2 *>(p)) : make_float2(0.f, 0.f);
                ov[j][0] = x.x;
                ov[j][1] = x.y;
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float f = q0 + j < n ? wq[q0 + j] : 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] += f * ov[j][e];
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) store_as(out + lane * E + e, W > 0.f ? acc[e] / W : 0.f);
    if (lse2 && lane == 0) *lse2 = W > 0.f ? M + log2f(W) : -INFINITY;
    __syncwarp();
}

}  // namespace
}  // namespace ikv
