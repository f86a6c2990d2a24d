// Top-k selection and gate weights of one token by one warp (Sec. 3.2: each token activates
// K of the E experts).  Lane l holds logits l, l+32, ...; selection runs k rounds of a warp
// arg-max on the raw fp32 logits (ties: lower expert index), so it is exact and independent
// of the score function.  Scores use expf.
#pragma once
#include <float.h>

#include "common.cuh"

namespace moe {

// Floats as unsigned integers of the same order (for the warp's integer reductions): never 0, and
// -0 becomes +0, so that equal floats have equal keys.
__device__ __forceinline__ uint32_t order_key(float v)
{
    const uint32_t u = __float_as_uint(v + 0.f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float order_value(uint32_t key)
{
    return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}

// All 32 lanes call it with the token's logits z[0..E).  On return lane j < k holds the j-th
// selected expert in sel_i and its gate weight (already multiplied by routed_scale) in sel_w.
// A chain of latencies for a few tokens, so a round is two integer warp reductions (largest key,
// then lowest index that holds it) instead of ten dependent shuffles.  Layer, with the grouping of
// up to 32 assignments shortened as well: tiny shape T = 16 22.4 -> 21.3 us, Qwen1.5 shape T = 1
// 38.1 -> 36.9, T = 5 68.5 -> 67.7.
template <int VPL>
__device__ __forceinline__ void warp_route_topk(const float *__restrict__ z, int E, int k,
                                                int score_fn, int renormalize, float routed_scale,
                                                int lane, int &sel_i, float &sel_w)
{
    float v[VPL];
    uint32_t key[VPL];  // 0: not (or no longer) to be selected
    uint32_t kmax = 0;
#pragma unroll
    for (int i = 0; i < VPL; ++i) {
        const int e = lane + 32 * i;
        v[i] = e < E ? z[e] : -FLT_MAX;
        if (!(v[i] == v[i]))
            v[i] = -FLT_MAX;  // NaN (outside the contract) ranks lowest
        key[i] = e < E ? order_key(v[i]) : 0u;
        kmax = max(kmax, key[i]);
    }
    // (at least -FLT_MAX, also where every logit is -infinity)
    const float vmax = fmaxf(order_value(__reduce_max_sync(0xffffffffu, kmax)), -FLT_MAX);
    float denom = 1.f;
    if (score_fn == MOE_SCORE_SOFTMAX) {
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < VPL; ++i)
            if (lane + 32 * i < E)
                sum += expf(v[i] - vmax);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            sum += __shfl_xor_sync(0xffffffffu, sum, off);
        denom = sum;
    }

    float sel_v = 0.f;
    sel_i = 0;
    for (int j = 0; j < k; ++j) {
        uint32_t bk = 0;
        int bi = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < VPL; ++i)
            if (key[i] > bk) {
                bk = key[i];
                bi = lane + 32 * i;
            }
        const uint32_t top = __reduce_max_sync(0xffffffffu, bk);
        bi = __reduce_min_sync(0xffffffffu, bk == top ? bi : 0x7fffffff);
#pragma unroll
        for (int i = 0; i < VPL; ++i)
            if (bi == lane + 32 * i)
                key[i] = 0u;
        if (lane == j) {
            sel_v = order_value(top);
            sel_i = bi;
        }
    }
    float p = 0.f;
    if (lane < k) {
        if (score_fn == MOE_SCORE_SOFTMAX)
            p = expf(sel_v - vmax) / denom;
        else
            p = 1.0f / (1.0f + expf(-sel_v));
    }
    if (renormalize) {
        float s = p;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, off);
        p = p / s;
    }
    sel_w = p * routed_scale;
}

}  // namespace moe
