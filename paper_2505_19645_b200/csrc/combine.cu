// Gate-weighted combine: out[t] = sum_j w[t,j] * y[inv_perm[t*K+j]] + s[t] * shared_y[t]
// (y and shared_y may arrive as partial planes, one per k chunk of the down projection).
// Gather form (each output row is summed in slot order by one owner), so the result does
// not depend on scheduling; 128-bit loads and stores.
#include "common.cuh"

namespace moe {

constexpr int CB_THREADS = 256;
constexpr int MOE_MAX_SHARED_PARTS = 8;  // k chunks of the shared expert's down pass, at most

__device__ __forceinline__ void accumulate8(float (&acc)[8], float w, const uint4 &v)
{
    acc[0] = fmaf(w, bf16_lo(v.x), acc[0]);
    acc[1] = fmaf(w, bf16_hi(v.x), acc[1]);
    acc[2] = fmaf(w, bf16_lo(v.y), acc[2]);
    acc[3] = fmaf(w, bf16_hi(v.y), acc[3]);
    acc[4] = fmaf(w, bf16_lo(v.z), acc[4]);
    acc[5] = fmaf(w, bf16_hi(v.z), acc[5]);
    acc[6] = fmaf(w, bf16_lo(v.w), acc[6]);
    acc[7] = fmaf(w, bf16_hi(v.w), acc[7]);
}

// Eight consecutive values of a row as they are stored: bf16, or floats for calls of a few tokens.
template <bool F32>
struct Row8;
template <>
struct Row8<false> {
    uint4 v;
    __device__ __forceinline__ void load(const void *base, size_t at)
    {
        v = *reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(base) + at);
    }
    __device__ __forceinline__ void add(float (&acc)[8], float w) const { accumulate8(acc, w, v); }
};
template <>
struct Row8<true> {
    float4 lo, hi;
    __device__ __forceinline__ void load(const void *base, size_t at)
    {
        const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(base) + at);
        lo = p[0];
        hi = p[1];
    }
    __device__ __forceinline__ void add(float (&acc)[8], float w) const
    {
        acc[0] = fmaf(w, lo.x, acc[0]);
        acc[1] = fmaf(w, lo.y, acc[1]);
        acc[2] = fmaf(w, lo.z, acc[2]);
        acc[3] = fmaf(w, lo.w, acc[3]);
        acc[4] = fmaf(w, hi.x, acc[4]);
        acc[5] = fmaf(w, hi.y, acc[5]);
        acc[6] = fmaf(w, hi.z, acc[6]);
        acc[7] = fmaf(w, hi.w, acc[7]);
    }
};

// KP: top_k rounded up to 2, 4, 8 or 16 -- the arrays of row pieces in flight are sized by it,
// so that a top-2 or top-4 layer keeps its registers (and its occupancy).
template <int KP, bool F32>
__global__ void __launch_bounds__(CB_THREADS, F32 ? 1 : (KP <= 2 ? 4 : (KP <= 4 ? 3 : (KP <= 8 ? 2 : 1))))
combine_kernel(const void *__restrict__ y, int routed_parts,
               const int32_t *__restrict__ inv_perm, const float *__restrict__ topk_w,
               const void *__restrict__ shared_y, int shared_parts,
               const float *__restrict__ shared_scale, int T, int H, int k,
               __nv_bfloat16 *__restrict__ out)
{
    griddep_launch();
    griddep_wait();  // y and shared_y come from the preceding kernel
    const int vec_per_row = H >> 3;
    const size_t plane = (size_t)T * k * H;
    // A thread's pieces lie gridDim x CB_THREADS apart; their (token, column) advance by additions (no
    // 64-bit division per piece), and the positions of the next piece are requested while the rows of
    // the current one are in flight; the weights too where registers are left for them (one CTA per SM:
    // top-16 of 7168 columns, T = 3072 172.0 -> 167.4 us), else they come with the rows (their registers
    // spilled at eight rows: top-8 of 7168 columns, T = 1280 38.8 -> 37.7).  Bound by loads in flight:
    // 2 CTAs of 256 threads per SM with eight 16-byte row pieces each.  A division per piece and no
    // positions ahead -> this, alone, inputs larger than L2, us: top-8 of 7168 columns T = 3072
    // 94.7 -> 86.8 (5.1 TB/s), T = 640 23.3 -> 20.6; of 3584, T = 1280 23.3 -> 20.6; top-2 of 3584,
    // T = 1280 9.7 -> 8.9; top-4 of 2048, T = 640 5.8 -> 5.4; three CTAs per SM at eight rows spill.
    constexpr bool WEIGHTS_AHEAD = KP > 8 && !F32;
    const unsigned step = gridDim.x * CB_THREADS, step_t = step / vec_per_row;
    const unsigned step_v = step - step_t * vec_per_row;
    const unsigned first = blockIdx.x * CB_THREADS + threadIdx.x;
    int t = (int)(first / vec_per_row), v8 = (int)(first - (unsigned)t * vec_per_row);
    int rows[KP];
    float wts[WEIGHTS_AHEAD ? KP : 1];
    auto weight = [&](int tok, int j) { return j < k ? topk_w[(size_t)tok * k + j] : 0.f; };
    auto fetch = [&](int tok) {
#pragma unroll
        for (int j = 0; j < KP; ++j) {
            rows[j] = j < k ? inv_perm[(size_t)tok * k + j] : 0;
            if constexpr (WEIGHTS_AHEAD)
                wts[j] = weight(tok, j);
        }
    };
    if (t < T)
        fetch(t);
    while (t < T) {
        const int h = v8 << 3;
        const float s = shared_y && shared_scale ? shared_scale[t] : 1.0f;
        // the shared expert's planes, four at a time, requested before the routed rows are used
        Row8<F32> sv[4];
        const int sp0 = shared_y ? (shared_parts < 4 ? shared_parts : 4) : 0;
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if (p < sp0)
                sv[p].load(shared_y, ((size_t)p * T + t) * H + h);
        float acc[8], cur_w[KP];
        const int cur_t = t;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            acc[q] = 0.f;
#pragma unroll
        for (int j = 0; j < KP; ++j)
            cur_w[j] = WEIGHTS_AHEAD ? wts[WEIGHTS_AHEAD ? j : 0] : weight(cur_t, j);
        t += (int)step_t;
        v8 += (int)step_v;
        if (v8 >= vec_per_row) {
            v8 -= vec_per_row;
            ++t;
        }
        for (int part = 0; part < routed_parts; ++part) {
            Row8<F32> v[KP];
#pragma unroll
            for (int j = 0; j < KP; ++j)
                if (j < k)
                    v[j].load(y, (size_t)part * plane + (size_t)rows[j] * H + h);
            if (part == routed_parts - 1 && t < T && t != cur_t)
                fetch(t);
#pragma unroll
            for (int j = 0; j < KP; ++j)
                if (j < k)
                    v[j].add(acc, cur_w[j]);
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if (p < sp0)
                sv[p].add(acc, s);
        if (shared_y && shared_parts > 4) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (4 + p < shared_parts)
                    sv[p].load(shared_y, ((size_t)(4 + p) * T + cur_t) * H + h);
#pragma unroll
            for (int p = 0; p < 4; ++p)
                if (4 + p < shared_parts)
                    sv[p].add(acc, s);
        }
        uint4 o;
        __nv_bfloat162 p;
        p = __floats2bfloat162_rn(acc[0], acc[1]);
        o.x = *reinterpret_cast<uint32_t *>(&p);
        p = __floats2bfloat162_rn(acc[2], acc[3]);
        o.y = *reinterpret_cast<uint32_t *>(&p);
        p = __floats2bfloat162_rn(acc[4], acc[5]);
        o.z = *reinterpret_cast<uint32_t *>(&p);
        p = __floats2bfloat162_rn(acc[6], acc[7]);
        o.w = *reinterpret_cast<uint32_t *>(&p);
        *reinterpret_cast<uint4 *>(out + (size_t)cur_t * H + h) = o;
    }
}

cudaError_t launch_combine(const moe_config_t &c, const __nv_bfloat16 *y, int routed_parts,
                           const int32_t *inv_perm, const float *topk_w,
                           const __nv_bfloat16 *shared_y, int shared_parts,
                           const float *shared_scale, int T, __nv_bfloat16 *out, cudaStream_t s, bool f32)
{
    if (shared_parts > MOE_MAX_SHARED_PARTS)
        return cudaErrorInvalidValue;
    const size_t total = (size_t)T * (c.hidden >> 3);
    size_t blocks = (total + CB_THREADS - 1) / CB_THREADS;
    // as many CTAs as are resident at once (see the launch bounds): every thread has the same number
    // of pieces or one less
    const int per_sm = f32 ? 1 : c.top_k <= 2 ? 4 : c.top_k <= 4 ? 3 : c.top_k <= 8 ? 2 : 1;
    const size_t cap = (size_t)sm_count() * per_sm;
    if (blocks > cap)
        blocks = cap;
#define MOE_CB_LAUNCH(KP)                                                                        \
    return f32 ? launch_pdl(combine_kernel<KP, true>, dim3((unsigned)blocks), dim3(CB_THREADS), 0, s, y, \
                            routed_parts, inv_perm, topk_w, shared_y, shared_parts, shared_scale, T, \
                            c.hidden, c.top_k, out)                                                  \
               : launch_pdl(combine_kernel<KP, false>, dim3((unsigned)blocks), dim3(CB_THREADS), 0, s, y, \
                            routed_parts, inv_perm, topk_w, shared_y, shared_parts, shared_scale, T, \
                            c.hidden, c.top_k, out)
    if (c.top_k <= 2)
        MOE_CB_LAUNCH(2);
    if (c.top_k <= 4)
        MOE_CB_LAUNCH(4);
    if (c.top_k <= 8)
        MOE_CB_LAUNCH(8);
    MOE_CB_LAUNCH(16);
#undef MOE_CB_LAUNCH
}

}  // namespace moe
