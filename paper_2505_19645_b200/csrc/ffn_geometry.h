// How the FFN kernels are shaped for a call (host only): segment size, CTA pairs, rings.  The host
// never sees the routing result; everything follows from the configuration and the token count.
#pragma once
#include <math.h>

#include "ffn_walk.cuh"
#include "moe_verify.h"

namespace moe {

int sm_count();  // SMs of the current device

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

inline int ffn_grid() { return sm_count(); }

// What pulls work items: a CTA, or a pair of CTAs whose tiles are twice as high.
struct FfnWorkers {
    int ctas, count;
};
inline FfnWorkers ffn_workers(const moe_config_t &c, int T)
{
    const int ctas = ffn_pairs(c, T) ? 2 : 1;
    return FfnWorkers{ctas, ffn_grid() / ctas};
}

// Weight rows of a routed tile per CTA in the two passes.  Full height (128 features with their gate
// and up rows, or 256 down rows) streams best, but where that gives few items, SMs stand idle while
// others pull a whole tile at what a single SM takes in (about 65 GB/s: four microseconds for
// 256 x 512).  Tiles of half the height are worth it while the items of BOTH passes fit the workers at
// once: the down pass's CTAs start on the SMs that the gate/up pass leaves alone, and its prologue
// shows where none are left.  Beyond that only a tile that streams for long gains by it, while its own
// pass fits.
//
// Measured on twenty small shapes (1 to 64 experts, hidden 256 to 4096) at T = 5 to 640 and on calls
// of one to four tokens, full height in both passes -> this: 3 % less in the mean, at best 11 %,
// nowhere more than 2.8 % more; tiny shape T = 16 18.6 -> 17.6 us, T = 128 22.9 -> 21.6.  With the
// height halved down to 64 rows while each pass alone fits the workers, 16 experts of 512 x 512
// T = 16 22.2 -> 25.6, T = 160 27.7 -> 32.2.  Down tiles of 64 rows: within 2 % of 128 where there is
// room, up to 40 % slower where there is not.
constexpr int FF_LONG_UP = 4096, FF_LONG_DOWN = 1024;  // reduction of a tile that streams for long
struct TileRows {
    int up, down;
};
inline TileRows routed_tile_rows(const moe_config_t &c, int T, int routed_parts)
{
    const FfnWorkers wk = ffn_workers(c, T);
    const double n_act = expected_active_experts(c.n_experts, c.top_k, T);
    const double segs = ceil(n_act) * ceil((double)T * c.top_k / n_act / segment_rows(c, T));
    auto up_items = [&](int h) { return segs * ((c.inter + h * wk.ctas - 1) / (h * wk.ctas)); };
    auto down_items = [&](int h) {
        return segs * routed_parts * ((c.hidden + h * wk.ctas - 1) / (h * wk.ctas));
    };
    const bool low_down = up_items(128) + down_items(128) <= wk.count ||
                          (c.inter / routed_parts >= FF_LONG_DOWN && down_items(128) <= wk.count);
    const int down = low_down ? 128 : 256;
    const bool low_up = up_items(64) + down_items(down) <= wk.count ||
                        (c.hidden >= FF_LONG_UP && up_items(64) <= wk.count);
    return TileRows{low_up ? 64 : 128, down};
}

// CTAs per SM of the row gather.  An FFN CTA does not start on an SM while a CTA of another kernel is
// resident there (measured, whatever their shared-memory and register needs), so until the gather has
// finished the gate/up pass runs its shared-expert tiles only on the SMs the gather leaves alone.  Up
// to 16 MB of rows it therefore runs as one CTA per SM at most (the hardware places them on about half
// of the SMs; fewer, larger CTAs made the gather itself too slow); a large gather needs every SM's full
// thread count.  Layer beyond 8192 assignments, eight CTAs per SM -> one, 16 experts top-4 of 256 and a
// shared one of 512, T = 2080, us: hidden 128 48.4 -> 45.4, 512 65.3 -> 62.8, 992 80.3 -> 77.8;
// 64 experts top-8, T = 2048, within 1 %.  Without a shared expert nothing could start early (8 experts
// top-2 of 512, T = 4200, hidden 768: 67.4 -> 70.3).
inline int gather_ctas_per_sm(const moe_config_t &c, int T, bool with_shared)
{
    return with_shared && (size_t)T * c.top_k * c.hidden * 2 <= (16u << 20) ? 1 : 8;
}

}  // namespace moe
