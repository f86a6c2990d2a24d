// How the FFN kernels are shaped for a call (host only): segment size, CTA pairs, rings.  The host
// never sees the routing result; everything follows from the configuration and the token count.
#pragma once
#include <math.h>

#include "ffn_walk.cuh"
#include "moe_verify.h"

namespace moe {

// Test hooks, read once per process.  MOE_FF_WIDE: 0 / 1 forces the ring geometry with segments of
// 128 / 256 rows, -1 (unset) leaves the choice to segment_rows().
int geometry_override();
// MOE_FF_PAIR: 1 runs the FFN kernels on CTA pairs in every call.
bool pairs_forced();

// Expected number of activated experts for T tokens (Eq. N(t): E(1 - (1 - K/E)^T)); the host
// never sees the routing result, so it sizes rings and shared tiles from the expectation.
inline double expected_active_experts(int E, int k, int T)
{
    return E * (1.0 - pow(1.0 - (double)k / E, (double)T));
}

// Segment size of a call (the N limit of its tensor-core instructions).  Groups in the hundreds
// of rows want the contraction geometry: segments of 256 rows, so that a weight tile is fetched
// once per 256 tokens and the instruction runs at its full rate.  Small groups want the
// streaming geometry (segments of 128 rows, 64 KB weight slots, double-buffered accumulators).
// The host never sees the routing result, so it decides on the expected rows per group -- and on
// the shared expert, whose group is all T tokens: where its weights are a large part of the
// layer's, every extra segment is another pass over them through L2.
inline int segment_rows(const moe_config_t &c, int T)
{
    const int force = geometry_override();
    if (force >= 0)
        return force == 1 ? FF_SEG_WIDE : FF_SEG;
    if (T <= FF_SEG)
        return FF_SEG;
    // measured cross-over: about 112 expected rows per group (most groups then exceed one
    // 128-row segment), or a shared expert several times an expert's size
    const double rows_per_group = (double)T * c.top_k / expected_active_experts(c.n_experts, c.top_k, T);
    if (rows_per_group > 0.875 * FF_SEG)
        return FF_SEG_WIDE;
    return c.shared_inter >= 6 * c.inter ? FF_SEG_WIDE : FF_SEG;
}

// Up to 128 tokens no group of the layer has more than one 128-row segment and the token ring
// can be 32 KB, which leaves room for a third weight slot (worth 3-4 % of the layer) --
// provided the entries stay within half of the ring, i.e. 64 rows: always so up to 64 tokens;
// between 65 and 128 tokens only while the routed groups are expected to be small (a larger
// group still works, its rows are then not fetched ahead), and the shared expert's rows are
// then cut into two 64-row segments.
inline bool small_token_ring(const moe_config_t &c, int T)
{
    if (T <= FF_SEG / 2)
        return true;
    if (T > FF_SEG)
        return false;
    // (a mean of up to a quarter of a segment: the largest group then stays within a half)
    return (double)T * c.top_k / expected_active_experts(c.n_experts, c.top_k, T) <= FF_SEG / 4 + 0.5;
}

// Token rows per segment of the shared expert (see small_token_ring).
inline int shared_segment_rows(const moe_config_t &c, int T)
{
    if (T > FF_SEG / 2 && small_token_ring(c, T))
        return FF_SEG / 2;
    return segment_rows(c, T);
}

// Whether the FFN kernels of a call run on CTA pairs: always in the contraction geometry (see the
// top of the file), in the streaming one beyond 128 tokens.  There a pair's token entries are half
// as large, so that three weight slots fit where a single CTA has two (96 KB of token ring for
// segments of 128 rows; the kernels' single-CTA instances are built for the streaming geometry
// alone).  Layer on single CTAs -> pairs, when both could be chosen: DeepSeek-V3 shape T = 256 3367 -> 3287 us,
// T = 1024 3647 -> 3560, T = 2048 4075 -> 3944, T = 3072 4428 -> 4374; Mixtral shape T = 192
// 488 -> 474, T = 384 537 -> 527; Qwen1.5 shape T = 192 to 640 within 1 %.  Up to 128 tokens the
// token rows are a small part of what an SM loads, single CTAs have three slots too, and a pair
// waits for the slower of its two streams (DeepSeek-V3 shape T = 128 3172 on single CTAs, 3248 on
// pairs; Mixtral shape T = 80 443 and 450).
inline bool ffn_pairs(const moe_config_t &c, int T)
{
    return segment_rows(c, T) > FF_SEG || T > FF_SEG || pairs_forced();
}

// Ring geometry.  Streaming: two k boxes per weight slot (64 KB for a full tile: every row is
// fetched in 256 contiguous bytes, which both HBM and L2 serve markedly faster than 128); the
// token ring holds two entries of the largest possible segment on CTA pairs and while no group
// can exceed 64 rows (32 KB, three weight slots), three 128-row entries otherwise (96 KB, two
// slots).  (One k box per slot, five slots, measured 3-4 % slower on pairs as well.)
// Contraction: pairs, one k box per slot and per entry, four entries of half a 256-row segment
// (64 KB), five slots.
inline void ffn_geometry(const moe_config_t &c, int T, FfnArgs &a)
{
    a.seg_rows = segment_rows(c, T);
    const bool wide = a.seg_rows > FF_SEG;
    a.kboxes = wide ? 1 : 2;
    a.acc_sets = wide ? 1 : 2;
    a.w_slot_bytes = 256 * 128 * a.kboxes;  // a full tile: 256 rows per k box
    // (a CTA of a pair holds half of a segment's rows: entries of at most 16 KB in both geometries)
    const int x_ring_bytes = wide ? 64 * 1024
                             : ffn_pairs(c, T) || small_token_ring(c, T) ? 32 * 1024 : 96 * 1024;
    a.x_units = x_ring_bytes / FF_X_UNIT;
    const int avail = FF_SMEM_LIMIT - 1024 - 512;  // alignment slack, static shared memory
    int ns = (avail - x_ring_bytes) / a.w_slot_bytes;
    if (ns > FF_STEPS)
        ns = FF_STEPS;
    a.n_w_slots = ns;
    a.shared_seg = shared_segment_rows(c, T);
}

}  // namespace moe
