// The work items of the FFN kernels: how the workers of the persistent grid divide the shared
// expert's units and claim the routed work, and where the token ring's entries lie.  It uses the
// barrier, cluster and warp primitives by the names of tc_ptx.cuh, which the includer provides
// first: the kernels' own, or a host program's, which runs the same walk on threads.
#pragma once
#include "plan.h"

namespace moe {

constexpr int FF_EPI_WARPS = 8;
constexpr int FF_THREADS = 32 * (3 + FF_EPI_WARPS);
constexpr int FF_STEPS = 8;  // k steps in flight: barrier pairs, token-ring entries, weight slots at most
static_assert(SEG_TOKENS == 128, "n_segments() divides by shifts");
constexpr int FF_SEG = SEG_TOKENS;        // token rows per segment in the streaming geometry
constexpr int FF_SEG_WIDE = 2 * SEG_TOKENS;  // ... in the contraction geometry (the MMA's N limit)
constexpr int FF_TMEM_COLS = 512;
constexpr int FF_SMEM_LIMIT = 227 * 1024;
constexpr int FF_X_UNIT = 2048;  // token ring unit: 16 rows x 128 bytes
constexpr int FF_HEIGHTS = 4;    // TMA box heights for weight tiles: 128, 64, 32, 16 rows

struct FfnArgs {
    int rows[2];   // output features per group kind (0 routed, 1 shared), multiples of 16
    int K[2];      // reduction length per group kind
    __nv_bfloat16 *out[2];
    int out_ld[2];
    int f32_out;   // down pass: out[] are float planes (same element offsets), see f32_outputs
    const int32_t *plan_header;  // [0] = [1] = number of segments
    const Segment *seg;
    const PairEntry *pairs;      // one entry per segment, with its group
    int max_pairs;               // capacity of the table
    int32_t *claim_counter;      // grid-wide: next unclaimed routed position / item of this pass
    int32_t *done[2];            // per segment of each group kind: 16-column units of h finished
                                 // by the gate/up pass, summed over its eight epilogue warps
    int first_fixed;             // round-robin mode: every worker's first item is fixed
    int round_robin;             // routed work dealt as (pair, tile) items instead of ranges
    int32_t *status;
    int T;             // token rows (the shared expert's group)
    int with_shared;   // shared expert present in this launch
    int shared_ksplit;   // k chunks of the shared expert's reduction (down pass; 1 = whole K):
                         // chunk s covers [s * shared_kchunk, ...) and writes its partial sums
                         // to out[1] + s * shared_part_stride
    int shared_kchunk;   // multiple of 128
    long long shared_part_stride;  // elements
    int routed_ksplit;   // the same for the routed groups (round-robin mode of the down pass only)
    int routed_kchunk;
    long long routed_part_stride;
    int shared_tiles;  // tiles of the shared expert's rows; (tile, k chunk, segment) units are dealt
                       // round-robin to the CTAs; the first (units % tiles) tiles have one
                       // 16-row unit more
    int max_tile;      // weight rows per tile and CTA: 128 (gate + up stacked) or 256 (down)
    int kboxes;        // 64-element k boxes per weight slot
    int w_slot_bytes;  // capacity of a weight slot
    int n_w_slots;
    int x_units;       // token ring size in FF_X_UNIT units
    int wait_us;       // limit of every wait inside the kernel, microseconds
    int seg_rows;      // token rows per segment of the routed groups (as in the plan): 128 or 256
    int shared_seg;    // token rows per segment of the shared expert: seg_rows, or 64 for
                       // 64 < T <= 128 with the small token ring (no entry beyond 16 KB)
    int acc_sets;      // accumulator sets in TMEM: 2 (segments up to 128 rows: a set is 2 x 128
                       // columns) or 1 (up to 256 rows: 2 x 256 columns)
};

// One work item: one segment of token rows of a group against one tile of its weight rows.
struct Item {
    int grp;     // 0 routed, 1 shared
    int expert;  // routed expert id (0 for the shared expert)
    int f0;      // first output feature (weight row inside the expert), multiple of 16
    int h;       // output features of the tile, multiple of 16 (pair: of 32, half of them per CTA)
    int row0;    // first token row (sorted row for routed groups, token for the shared expert)
    int n;       // token rows, 1..seg_rows
    int seg;     // index of the segment's progress counter (plan index; shared: segment number)
    int w_once;  // the tile's weights are read by this item only
    int k0, k1;  // reduction range [k0, k1)
    long long out_off;  // element offset of this item's output plane (k chunk) in out[grp]
};

// Hand-over of the routed work a CTA claims at run time.  One thread of the CTA (the weight
// producer) claims chunks from a grid-wide counter and publishes them in a small ring; the
// other roles read the same sequence, so all roles walk identical items.
constexpr int FF_CLAIMS = 4;      // ring entries
// token producer, MMA issuer, epilogue warps; in the second CTA of a pair the weight producer
// reads as well and nothing is issued
constexpr int FF_CLAIM_READERS = 2 + FF_EPI_WARPS;

constexpr int FF_CLAIM_WORDS = 8;  // lo, hi, and (round-robin mode) the item's group, decoded
struct ClaimRing {
    int *data;                 // shared memory [FF_CLAIMS][FF_CLAIM_WORDS]
    uint32_t full0, empty0;    // shared addresses of the barrier arrays [FF_CLAIMS]
    volatile int *abort_flag;
    int32_t *status;
    // a pair's ring: the leader claims for both CTAs and writes both copies of an entry; the
    // readers of both CTAs arrive on the leader's empty barriers (cluster addresses)
    uint32_t peer_data, peer_full0, leader_empty0;
};

// Walks the items of one CTA, in every lane of the role's warp: its units of the shared expert first (dealt round-robin: they
// depend on nothing the layer computes), then chunks of the routed groups' work, claimed from
// a grid-wide counter so that a CTA that is late or slow simply takes less.  The routed part
// needs the segment plan, which the preceding kernels write: next() calls
// griddepcontrol.wait once before it touches the plan (or before reporting the end).
//
// Routed work, range mode: positions (16 rows of one group for one of its segments, groups
// laid end to end); a chunk is a run of positions whose ends are moved to tile boundaries, its
// length shrinks as the work runs out (a third of the remaining per-CTA share, at least one
// tile).  Round-robin mode: a chunk is one (segment, tile, k chunk) item; consecutive items are
// the tiles of one segment, which then run on many CTAs at once and share the segment's token
// rows in L2.
// Rows per segment of a group of n rows cut into nseg segments: equal shares rounded up to the
// 16-row unit of the token boxes (never more than the segment limit, since nseg = ceil(n /
// limit)).  Equal shares instead of "full segments and a remainder": the instruction time
// follows the rows of a segment with a floor of about 64 rows, so 320 rows cost less as
// 160 + 160 than as 256 + 64.
__device__ __forceinline__ int balanced_segment_rows(int n, int nseg)
{
    return nseg == 1 ? (n + 15) & ~15 : (((n + nseg - 1) / nseg) + 15) & ~15;
}

// PAIR: the worker is a CTA pair that walks the items together, each CTA computing half of a
// tile's features; row units are then 32 weight rows, so that the halves are whole 16-row units.
template <bool PAIR>
struct ItemWalk {
    static constexpr int USH = PAIR ? 5 : 4;  // log2 of the weight rows of a unit
    const FfnArgs &a;
    const ClaimRing &ring;
    const bool claimer;    // this warp's first lane claims; all others follow the ring
    const bool lead;       // first lane: claims, or arrives on the ring's barriers for its role
    const int max_units;
    const int worker, workers;
    int n_claims;
    // shared expert: units (tile, k chunk, segment) sj, sj + grid, ...
    int sj, Us, s_base, s_rem, nseg_s, s_units;
    // routed groups: current chunk from (fs, u) to (fs_hi, u_hi); fs = plan index of a
    // group's first segment
    int R0, nseg_total, fs, u, fs_hi, u_hi;
    long long P;
    int ntiles;
    bool synced, group_loaded, have_chunk, finished, end_published;
    int n_pub;  // claimer: chunks published so far
    int4 pair_group;  // claimer: the plan entry looked up last
    int pair_seg;
    // current group and tile
    Segment sg;
    int g_nseg, g_u_end;
    bool have_tile;
    int t_grp, t_expert, t_u0, t_h, t_row0, t_n, t_s, t_s_end, t_seg0, t_seg_rows;
    bool t_once;  // the tile's weights are read by this pass over it only
    int t_k0, t_k1;
    long long t_out_off;

    __device__ ItemWalk(const FfnArgs &args, const ClaimRing &r, bool is_claimer, bool already_synced)
        : a(args), ring(r), claimer(is_claimer), lead((threadIdx.x & 31) == 0),
          max_units(args.max_tile >> 4),  // a pair's tile is twice as high, as is its unit
          worker(PAIR ? blockIdx.x >> 1 : blockIdx.x), workers(PAIR ? gridDim.x >> 1 : gridDim.x),
          n_claims(0), synced(false), group_loaded(false), have_chunk(false), finished(false),
          end_published(false), n_pub(0),
          have_tile(false)
    {
        Us = a.with_shared ? a.rows[1] >> USH : 0;
        s_base = a.shared_tiles ? Us / a.shared_tiles : 0;
        s_rem = a.shared_tiles ? Us % a.shared_tiles : 0;
        sj = worker;
        nseg_s = (a.T + a.shared_seg - 1) / a.shared_seg;
        s_units = a.shared_tiles * a.shared_ksplit * nseg_s;
        R0 = a.rows[0] >> USH;
        nseg_total = fs = u = fs_hi = u_hi = 0;
        ntiles = (R0 + max_units - 1) / max_units;
        P = 0;
        if (already_synced)
            sync(false);
    }
    // segments of a group of n rows (seg_rows is 128 or 256)
    __device__ int n_segments(int n) const { return (n + a.seg_rows - 1) >> (a.seg_rows == SEG_TOKENS ? 7 : 8); }
    // position p -> (group, row unit rounded down to a tile boundary of the group)
    __device__ void boundary(long long p, int &fs_out, int &u_out) const
    {
        if (p >= P) {
            fs_out = nseg_total;
            u_out = 0;
            return;
        }
        const Segment s = a.seg[(int)(p / R0)];
        const int ns = n_segments(s.n);
        fs_out = s.first_seg;
        u_out = (int)((p - (long long)s.first_seg * R0) / ns) / max_units * max_units;
    }
    __device__ void sync(bool wait)
    {
        if (wait)
            griddep_wait();
        // (the entry of a fixed first item is requested with the header, not after it)
        const int4 hdr = *reinterpret_cast<const int4 *>(a.plan_header);
        if (claimer && lead && a.first_fixed)
            load_pair(min((workers - 1 - worker) / (ntiles * a.routed_ksplit), a.max_pairs - 1));
        nseg_total = hdr.x;
        P = a.round_robin ? (long long)hdr.y * ntiles * a.routed_ksplit : (long long)nseg_total * R0;
        synced = true;
    }
    // The plan's entry of a segment, with its group: one load level between a claim and its tile.
    __device__ void load_pair(int i)
    {
        const int4 *pe = reinterpret_cast<const int4 *>(a.pairs + i);
        pair_group = pe[0];
        pair_seg = pe[1].x;
    }
    // Claims the next chunk from the grid-wide counter (claimer only).  In round-robin mode
    // of the gate/up pass, whose workers all start together,
    // the first item of every worker is fixed -- item workers - 1 - worker, so that the workers
    // without a shared-expert tile (the high ones) take the first routed items -- and costs no
    // round trip to the counter; the counter hands out the items from `workers` on.  The workers
    // of the down pass start as the gate/up pass leaves their SMs, so all its items are handed
    // out in that order: with few items (8 at T = 16 on the tiny shape) a fixed share went to
    // the SMs that were busy longest (26.0 -> 22.4 us with the shorter path from the plan to the
    // first tile; Qwen1.5 shape T = 5 69.6 -> 68.5).
    __device__ void claim(int &lo, int &hi)
    {
        if (a.round_robin) {
            lo = !a.first_fixed  ? atomicAdd(a.claim_counter, 1)
                 : n_pub == 0 ? workers - 1 - worker
                              : workers + atomicAdd(a.claim_counter, 1);
            hi = lo + 1;
        } else {
            const long long left = P - peek(a.claim_counter);
            const long long guided = left / (3 * (long long)workers);
            const int size = (int)(guided > max_units ? guided : max_units);
            lo = atomicAdd(a.claim_counter, size);
            hi = (int)(lo + (long long)size < P ? lo + size : P);
        }
        if (lo >= P)
            lo = hi = -1;
    }
    // Claimer: claims one more chunk and publishes it in the ring (with its group looked up
    // in round-robin mode, so that the other roles need not go to global memory for it).
    __device__ bool publish_one()
    {
        const int slot = n_pub % FF_CLAIMS;
        const uint32_t par = (uint32_t)(n_pub / FF_CLAIMS) & 1u;
        int lo, hi, sidx = 0;
        Segment grp = sg;
        claim(lo, hi);
        if (lo >= 0 && a.round_robin) {
            if (n_pub > 0 || !a.first_fixed)
                load_pair(lo / (ntiles * a.routed_ksplit));
            sidx = pair_seg;
            grp.expert = pair_group.x;
            grp.row0 = pair_group.y;
            grp.n = pair_group.z;
            grp.first_seg = pair_group.w;
        }
        if (!mbar_wait<PAIR>(ring.empty0 + 8u * slot, par ^ 1u, ring.abort_flag, ring.status))
            return false;
        if (PAIR) {
            const uint32_t pe = ring.peer_data + slot * FF_CLAIM_WORDS * 4;
            st_cluster_v4(pe, lo, hi, sidx, grp.expert);
            st_cluster_v4(pe + 16, grp.row0, grp.n, grp.first_seg, 0);
            mbar_arrive_cluster(ring.peer_full0 + 8u * slot);
        }
        int *e = ring.data + slot * FF_CLAIM_WORDS;
        e[0] = lo;
        e[1] = hi;
        e[2] = sidx;
        e[3] = grp.expert;
        e[4] = grp.row0;
        e[5] = grp.n;
        e[6] = grp.first_seg;
        __threadfence_block();
        mbar_arrive(ring.full0 + 8u * slot);
        ++n_pub;
        if (lo < 0)
            end_published = true;
        return true;
    }
    // Next chunk [lo, hi) of the routed work; false when none is left (or on abort).  In
    // round-robin mode the chunk is one item and `grp` receives its group.  While plenty of
    // work is left the claimer publishes one chunk beyond the one it is about to work on, so
    // that every role knows its next item before it finishes the current one (near the end a
    // chunk held in reserve would starve another CTA).
    __device__ bool acquire(int &lo, int &hi, Segment &grp, int &sidx)
    {
        const int slot = n_claims % FF_CLAIMS;
        const uint32_t par = (uint32_t)(n_claims / FF_CLAIMS) & 1u;
        int *e = ring.data + slot * FF_CLAIM_WORDS;
        if (claimer) {
            bool published = true;
            while (lead) {
                // (the counter is only read where the answer can be yes)
                const long long ample = 4 * (long long)workers * (a.round_robin ? 1 : max_units);
                const bool plenty =
                    P > ample && P - peek(a.claim_counter) > ample;
                if (end_published || n_pub >= n_claims + (plenty ? 2 : 1))
                    break;
                if (!publish_one()) {
                    published = false;
                    break;
                }
            }
            if (!__all_sync(0xffffffffu, published))
                return false;
            // the first lane wrote the entry and no barrier stands between it and the others here
            // (a vote orders no memory); also: all lanes have read an entry before it is reused
            __syncwarp();
        } else {
            // (the lanes of a warp wait one by one: when a wait gives up, all leave together)
            const bool got = mbar_wait<PAIR>(ring.full0 + 8u * slot, par, ring.abort_flag, ring.status);
            if (!__all_sync(0xffffffffu, got))
                return false;
        }
        ++n_claims;
        lo = e[0];
        hi = e[1];
        sidx = e[2];
        grp.expert = e[3];
        grp.row0 = e[4];
        grp.n = e[5];
        grp.first_seg = e[6];
        if (!claimer) {
            __syncwarp();  // every lane has read the entry before it is released
            if (lead) {
                if (PAIR)
                    mbar_arrive_cluster(ring.leader_empty0 + 8u * slot);
                else
                    mbar_arrive(ring.empty0 + 8u * slot);
            }
        }
        return lo >= 0;
    }
    // false when this CTA has no further item
    __device__ bool next(Item &it)
    {
        for (;;) {
            if (have_tile) {
                if (t_s < t_s_end) {
                    it.grp = t_grp;
                    it.expert = t_expert;
                    it.f0 = t_u0 << USH;
                    it.h = t_h << USH;
                    it.row0 = t_row0 + t_s * t_seg_rows;
                    it.n = min(t_seg_rows, t_n - t_s * t_seg_rows);
                    it.seg = t_seg0 + t_s;
                    it.w_once = t_once;
                    it.k0 = t_k0;
                    it.k1 = t_k1;
                    it.out_off = t_out_off;
                    ++t_s;
                    return true;
                }
                have_tile = false;
            }
            if (sj < s_units) {  // next unit of the shared expert: (tile, k chunk, segment)
                const int tc = sj / nseg_s, q = sj - tc * nseg_s;
                const int tile = tc / a.shared_ksplit, chunk = tc - tile * a.shared_ksplit;
                t_k0 = chunk * a.shared_kchunk;
                t_k1 = min(a.K[1], t_k0 + a.shared_kchunk);
                t_out_off = chunk * a.shared_part_stride;
                t_u0 = tile * s_base + min(tile, s_rem);
                t_h = s_base + (tile < s_rem ? 1 : 0);
                t_grp = 1;
                t_expert = 0;
                t_row0 = 0;
                t_seg0 = 0;
                t_n = a.T;
                t_seg_rows = balanced_segment_rows(a.T, nseg_s);
                t_s = q;
                t_s_end = q + 1;
                t_once = nseg_s <= 1;
                sj += workers;
                have_tile = true;
                continue;
            }
            if (!synced)
                sync(true);
            if (finished)
                return false;
            if (!have_chunk) {
                int lo, hi, sidx;
                if (!acquire(lo, hi, sg, sidx)) {
                    finished = true;
                    return false;
                }
                if (a.round_robin) {
                    // one (segment, tile, k chunk) item
                    const int st = a.routed_ksplit == 1 ? lo : lo / a.routed_ksplit;
                    const int chunk = lo - st * a.routed_ksplit;
                    const int tile = st % ntiles;
                    g_nseg = n_segments(sg.n);
                    t_u0 = tile * max_units;
                    t_h = min(max_units, R0 - t_u0);
                    t_grp = 0;
                    t_expert = sg.expert;
                    t_row0 = sg.row0;
                    t_seg0 = sg.first_seg;
                    t_n = sg.n;
                    t_seg_rows = balanced_segment_rows(sg.n, g_nseg);
                    t_s = sidx - sg.first_seg;
                    t_s_end = t_s + 1;
                    t_once = g_nseg <= 1;
                    t_k0 = chunk * a.routed_kchunk;
                    t_k1 = min(a.K[0], t_k0 + a.routed_kchunk);
                    t_out_off = chunk * a.routed_part_stride;
                    have_tile = true;
                    continue;
                }
                boundary(lo, fs, u);
                boundary(hi, fs_hi, u_hi);
                group_loaded = false;
                have_chunk = true;
            }
            if (fs >= nseg_total || fs > fs_hi || (fs == fs_hi && u >= u_hi)) {
                have_chunk = false;  // chunk exhausted (or empty after rounding)
                continue;
            }
            if (!group_loaded) {
                sg = a.seg[fs];
                g_nseg = n_segments(sg.n);
                g_u_end = fs == fs_hi ? u_hi : R0;
                group_loaded = true;
            }
            if (u < g_u_end) {  // next tile of this group, all its segments
                t_h = min(max_units, g_u_end - u);
                t_grp = 0;
                t_expert = sg.expert;
                t_u0 = u;
                t_row0 = sg.row0;
                t_seg0 = sg.first_seg;
                t_n = sg.n;
                t_seg_rows = balanced_segment_rows(sg.n, g_nseg);
                t_s = 0;
                t_s_end = g_nseg;
                t_once = g_nseg <= 1;
                t_k0 = 0;
                t_k1 = a.K[0];
                t_out_off = 0;
                u += t_h;
                have_tile = true;
                continue;
            }
            fs += g_nseg;  // group done: on to the next one
            u = 0;
            group_loaded = false;
        }
    }
};

// Placement of the token-ring entries.  An entry takes `m` consecutive units and never wraps:
// when it does not fit before the end of the ring it starts at unit 0.  Producer and MMA
// issuer replay the same sequence of sizes, so they agree on every position.
struct XRingWalk {
    int units, cur, count;
    __device__ XRingWalk(int n_units) : units(n_units), cur(0), count(0) {}
    // returns the first unit of the next entry; `pad` = units skipped at the end of the ring
    __device__ int place(int m, int &pad)
    {
        pad = 0;
        if (cur + m > units) {
            pad = units - cur;  // may be 0 when the previous entry ended exactly at the end
            cur = 0;
        }
        const int at = cur;
        cur += m;
        ++count;
        return at;
    }
};

__device__ __forceinline__ int pieces16(int n) { return (n + 15) >> 4; }

// 16-row pieces of a segment's n token rows that one CTA loads: all, or half of them (rounded
// up) for each CTA of a pair.
template <bool PAIR>
__device__ __forceinline__ int token_pieces(int n)
{
    return PAIR ? (n + 31) >> 5 : pieces16(n);
}

}  // namespace moe
