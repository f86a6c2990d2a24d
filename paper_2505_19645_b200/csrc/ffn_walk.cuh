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
    const int32_t *plan_header;  // [0] = number of segments
    const Segment *seg;          // one entry per segment, with its group
    int max_seg;                 // capacity of the table
    int32_t *claim_counter;      // grid-wide: routed items of this pass claimed so far
    int32_t *done[2];            // per segment of each group kind: 16-column units of h finished
                                 // by the gate/up pass, summed over its eight epilogue warps
    int first_fixed;             // every worker's first routed item is fixed
    int32_t *status;
    int T;             // token rows (the shared expert's group)
    int with_shared;   // shared expert present in this launch
    int shared_ksplit;   // k chunks of the shared expert's reduction (down pass; 1 = whole K):
                         // chunk s covers [s * shared_kchunk, ...) and writes its partial sums
                         // to out[1] + s * shared_part_stride
    int shared_kchunk;   // multiple of 128
    long long shared_part_stride;  // elements
    int routed_ksplit;   // the same for the routed groups
    int routed_kchunk;
    long long routed_part_stride;
    int shared_tiles;  // tiles of the shared expert's rows; (tile, k chunk, segment) units are dealt
                       // round-robin to the CTAs; the first (units % tiles) tiles have one
                       // 16-row unit more
    int max_tile;      // most weight rows of a routed tile per CTA: 128 or 64 (gate + up stacked), 256
                       // or 128 (down), see routed_tile_rows(); the shared expert's tiles follow from
                       // shared_tiles and may be higher
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

// Hand-over of the routed work a worker claims at run time.  One thread (of the weight producer)
// claims items from a grid-wide counter and publishes them in a small ring; the other roles read
// the same sequence, so all roles walk identical items.
constexpr int FF_CLAIMS = 4;      // ring entries
// token producer, MMA issuer, epilogue warps; in the second CTA of a pair the weight producer
// reads as well and nothing is issued
constexpr int FF_CLAIM_READERS = 2 + FF_EPI_WARPS;

// An entry: the item's number (-1: none left), the plan index of its segment, and the segment's
// group (expert, row0, n, first_seg), so that the other roles need not look it up.
constexpr int FF_CLAIM_WORDS = 8;
struct ClaimRing {
    int *data;                 // shared memory [FF_CLAIMS][FF_CLAIM_WORDS]
    uint32_t full0, empty0;    // shared addresses of the barrier arrays [FF_CLAIMS]
    volatile int *abort_flag;
    int32_t *status;
    // a pair's ring: the leader claims for both CTAs and writes both copies of an entry; the
    // readers of both CTAs arrive on the leader's empty barriers (cluster addresses)
    uint32_t peer_data, peer_full0, leader_empty0;
};

// Rows per segment of a group of n rows cut into nseg segments: equal shares rounded up to the
// 16-row unit of the token boxes (never more than the segment limit, since nseg = ceil(n /
// limit)).  Equal shares instead of "full segments and a remainder": the instruction time
// follows the rows of a segment with a floor of about 64 rows, so 320 rows cost less as
// 160 + 160 than as 256 + 64.
__device__ __forceinline__ int balanced_segment_rows(int n, int nseg)
{
    return nseg == 1 ? (n + 15) & ~15 : (((n + nseg - 1) / nseg) + 15) & ~15;
}

// Walks the items of one worker, in every lane of the role's warp: its units of the shared expert
// first (dealt round-robin: they depend on nothing the layer computes), then the routed items it
// claims from a grid-wide counter, so that a worker that is late or slow simply takes less.  The
// routed part needs the segment plan, which the preceding kernels write: next() calls
// griddepcontrol.wait once before it touches the plan (or before reporting the end).
//
// A routed item is one (segment, tile, k chunk); consecutive items are the tiles of one segment,
// which then run on many SMs at once and share the segment's token rows in L2.  Ranges of
// consecutive tiles per worker instead, each "its" groups' rows, have uneven ends and coarse chunks:
// layer, ranges -> items, Qwen1.5 shape T = 77 180.2 -> 177.6 us, T = 128 189 -> 186, T = 192
// 199.4 -> 195.1, Qwen2 shape T = 64 589.6 -> 586.9, Mixtral and DeepSeek-V3 shapes equal.  (Items of
// half the tile height for the last round of every worker: 1-6 % slower.)
//
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
    int n_claims;  // items taken from the ring so far
    int n_pub;     // claimer: items published so far
    // shared expert: units (tile, k chunk, segment) sj, sj + workers, ...
    int sj, s_base, s_rem, nseg_s, s_units;
    // routed groups
    int R0, ntiles, n_items;  // row units of a group, tiles of a group, items of the pass
    bool synced, finished, end_published;
    Segment entry;  // claimer: the plan entry looked up last

    __device__ ItemWalk(const FfnArgs &args, const ClaimRing &r, bool is_claimer, bool already_synced)
        : a(args), ring(r), claimer(is_claimer), lead((threadIdx.x & 31) == 0),
          max_units(args.max_tile >> 4),  // a pair's tile is twice as high, as is its unit
          worker(PAIR ? blockIdx.x >> 1 : blockIdx.x), workers(PAIR ? gridDim.x >> 1 : gridDim.x),
          n_claims(0), n_pub(0), n_items(0), synced(false), finished(false), end_published(false)
    {
        const int Us = a.with_shared ? a.rows[1] >> USH : 0;
        s_base = a.shared_tiles ? Us / a.shared_tiles : 0;
        s_rem = a.shared_tiles ? Us % a.shared_tiles : 0;
        sj = worker;
        nseg_s = (a.T + a.shared_seg - 1) / a.shared_seg;
        s_units = a.shared_tiles * a.shared_ksplit * nseg_s;
        R0 = a.rows[0] >> USH;
        ntiles = (R0 + max_units - 1) / max_units;
        if (already_synced)
            sync(false);
    }
    // segments of a group of n rows (seg_rows is 128, or for pairs 256)
    __device__ int n_segments(int n) const
    {
        const int wide = PAIR && a.seg_rows != SEG_TOKENS;
        return (n + (SEG_TOKENS << wide) - 1) >> (7 + wide);
    }
    __device__ void sync(bool wait)
    {
        if (wait)
            griddep_wait();
        // (the entry of a fixed first item is requested with the header, not after it)
        const int4 hdr = *reinterpret_cast<const int4 *>(a.plan_header);
        if (claimer && lead && a.first_fixed)
            load_entry(min((workers - 1 - worker) / (ntiles * a.routed_ksplit), a.max_seg - 1));
        n_items = hdr.x * ntiles * a.routed_ksplit;
        synced = true;
    }
    // The plan's entry of a segment, with its group: one load level between a claim and its tile.
    __device__ void load_entry(int i)
    {
        const int4 *p = reinterpret_cast<const int4 *>(a.seg + i);
        const int4 group = p[0];
        entry.seg = p[1].x;
        entry.expert = group.x;
        entry.row0 = group.y;
        entry.n = group.z;
        entry.first_seg = group.w;
    }
    // Claims the next item (claimer only; -1: none left).  In the gate/up pass, whose workers all
    // start together, the first item of every worker is fixed -- item workers - 1 - worker, so
    // that the workers without a shared-expert tile (the high ones) take the first routed items --
    // and costs no round trip to the counter, which hands out the items from `workers` on.  The workers
    // of the down pass start as the gate/up pass leaves their SMs, so all its items are handed
    // out in that order: with few items (8 at T = 16 on the tiny shape) a fixed share went to
    // the SMs that were busy longest (26.0 -> 22.4 us with the shorter path from the plan to the
    // first tile; Qwen1.5 shape T = 5 69.6 -> 68.5).
    __device__ int claim()
    {
        const int i = !a.first_fixed ? atomicAdd(a.claim_counter, 1)
                      : n_pub == 0   ? workers - 1 - worker
                                     : workers + atomicAdd(a.claim_counter, 1);
        return i < n_items ? i : -1;
    }
    // Claimer: claims one more item and publishes it in the ring.
    __device__ bool publish_one()
    {
        const int slot = n_pub % FF_CLAIMS;
        const uint32_t par = (uint32_t)(n_pub / FF_CLAIMS) & 1u;
        const int item = claim();
        if (item >= 0 && (n_pub > 0 || !a.first_fixed))
            load_entry(item / (ntiles * a.routed_ksplit));
        if (!mbar_wait<PAIR>(ring.empty0 + 8u * slot, par ^ 1u, ring.abort_flag, ring.status))
            return false;
        if (PAIR) {
            const uint32_t pe = ring.peer_data + slot * FF_CLAIM_WORDS * 4;
            st_cluster_v4(pe, item, entry.seg, entry.expert, entry.row0);
            st_cluster_v4(pe + 16, entry.n, entry.first_seg, 0, 0);
            mbar_arrive_cluster(ring.peer_full0 + 8u * slot);
        }
        int *e = ring.data + slot * FF_CLAIM_WORDS;
        e[0] = item;
        e[1] = entry.seg;
        e[2] = entry.expert;
        e[3] = entry.row0;
        e[4] = entry.n;
        e[5] = entry.first_seg;
        __threadfence_block();
        mbar_arrive(ring.full0 + 8u * slot);
        ++n_pub;
        if (item < 0)
            end_published = true;
        return true;
    }
    // Next routed item and its segment; -1 when none is left (or on abort).  While plenty of work
    // is left the claimer publishes one item beyond the one it is about to work on, so that every
    // role knows its next item before it finishes the current one (near the end an item held in
    // reserve would starve another worker).
    __device__ int acquire(Segment &sg)
    {
        const int slot = n_claims % FF_CLAIMS;
        const uint32_t par = (uint32_t)(n_claims / FF_CLAIMS) & 1u;
        int *e = ring.data + slot * FF_CLAIM_WORDS;
        if (claimer) {
            bool published = true;
            while (lead) {
                // (the counter is only read where the answer can be yes)
                const int ample = 4 * workers;
                const bool plenty = n_items > ample && n_items - peek(a.claim_counter) > ample;
                if (end_published || n_pub >= n_claims + (plenty ? 2 : 1))
                    break;
                if (!publish_one()) {
                    published = false;
                    break;
                }
            }
            if (!__all_sync(0xffffffffu, published))
                return -1;
            // the first lane wrote the entry and no barrier stands between it and the others here
            // (a vote orders no memory); also: all lanes have read an entry before it is reused
            __syncwarp();
        } else {
            // (the lanes of a warp wait one by one: when a wait gives up, all leave together)
            const bool got = mbar_wait<PAIR>(ring.full0 + 8u * slot, par, ring.abort_flag, ring.status);
            if (!__all_sync(0xffffffffu, got))
                return -1;
        }
        ++n_claims;
        const int item = e[0];
        sg.seg = e[1];
        sg.expert = e[2];
        sg.row0 = e[3];
        sg.n = e[4];
        sg.first_seg = e[5];
        if (!claimer) {
            __syncwarp();  // every lane has read the entry before it is released
            if (lead) {
                if (PAIR)
                    mbar_arrive_cluster(ring.leader_empty0 + 8u * slot);
                else
                    mbar_arrive(ring.empty0 + 8u * slot);
            }
        }
        return item;
    }
    // false when this worker has no further item
    __device__ bool next(Item &it)
    {
        if (sj < s_units) {  // next unit of the shared expert: (tile, k chunk, segment)
            const int tc = sj / nseg_s, q = sj - tc * nseg_s;
            const int tile = tc / a.shared_ksplit, chunk = tc - tile * a.shared_ksplit;
            const int rows = balanced_segment_rows(a.T, nseg_s);
            it.grp = 1;
            it.expert = 0;
            it.f0 = (tile * s_base + min(tile, s_rem)) << USH;
            it.h = (s_base + (tile < s_rem ? 1 : 0)) << USH;
            it.row0 = q * rows;
            it.n = min(rows, a.T - q * rows);
            it.seg = q;
            it.w_once = nseg_s <= 1;
            it.k0 = chunk * a.shared_kchunk;
            it.k1 = min(a.K[1], it.k0 + a.shared_kchunk);
            it.out_off = chunk * a.shared_part_stride;
            sj += workers;
            return true;
        }
        if (!synced)
            sync(true);
        if (finished)
            return false;
        Segment sg;
        const int item = acquire(sg);
        if (item < 0) {
            finished = true;
            return false;
        }
        const int st = a.routed_ksplit == 1 ? item : item / a.routed_ksplit;
        const int chunk = item - st * a.routed_ksplit, tile = st % ntiles;
        const int u0 = tile * max_units, nseg = n_segments(sg.n), q = sg.seg - sg.first_seg;
        const int rows = balanced_segment_rows(sg.n, nseg);
        it.grp = 0;
        it.expert = sg.expert;
        it.f0 = u0 << USH;
        it.h = min(max_units, R0 - u0) << USH;
        it.row0 = sg.row0 + q * rows;
        it.n = min(rows, sg.n - q * rows);
        it.seg = sg.seg;
        it.w_once = nseg <= 1;
        it.k0 = chunk * a.routed_kchunk;
        it.k1 = min(a.K[0], it.k0 + a.routed_kchunk);
        it.out_off = chunk * a.routed_part_stride;
        return true;
    }
};

// Placement of the token-ring entries.  An entry takes `m` consecutive units and never wraps:
// when it does not fit before the end of the ring it starts at unit 0.  Producer and MMA
// issuer replay the same sequence of sizes, so they agree on every position.
struct XRingWalk {
    int units, cur, count, pad;
    __device__ XRingWalk(int n_units) : units(n_units), cur(0), count(0), pad(0) {}
    // returns the first unit of the next entry; `pad` = units skipped at the end of the ring
    __device__ int place(int m)
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

// The producer's side: which entries must have been consumed before the next one may be issued.
// place() an entry, wait for entry `released` and release() it while must_release(), then issue.
// `starts`: where each entry's rows begin, after its padding (an array of the caller's, so that the
// rest stays in registers).
struct TokenRing : XRingWalk {
    int released;            // entries known to have been consumed
    int v_cur, v_rel;        // virtual unit positions: issued up to / free up to
    int v_start, v_end;      // of the entry placed last
    __device__ TokenRing(int n_units) : XRingWalk(n_units), released(0), v_cur(0), v_rel(0), v_start(0), v_end(0) {}
    __device__ int place(int m)
    {
        const int at = XRingWalk::place(m);
        v_start = v_cur + pad;
        v_end = v_start + m;
        return at;
    }
    // the entry's units and its barrier pair must be free: everything before the oldest entry still
    // in use is, the padding in front of it included
    __device__ bool must_release() const
    {
        const int j = count - 1;
        return released < j && (j - released >= FF_STEPS || v_end - v_rel > units);
    }
    __device__ void release(const int (&starts)[FF_STEPS])
    {
        ++released;
        v_rel = released < count - 1 ? starts[released % FF_STEPS] : v_start;
    }
    __device__ void issued(int (&starts)[FF_STEPS])
    {
        starts[(count - 1) % FF_STEPS] = v_start;
        v_cur = v_end;
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
