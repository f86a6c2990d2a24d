// Expert FFN (gate/up + SwiGLU, and down projection) for every group size: the activated
// experts' weights are streamed from HBM exactly once by TMA through a ring of shared-memory
// slots and contracted on the tensor cores (tcgen05.mma, fp32 accumulators in TMEM).
//
// Orientation.  Measured on this part, one tcgen05.mma kind::f16 of shape M x N x 16 occupies
// the tensor pipe for max(48.5, N / 2) cycles, whatever M in {64, 128} is and whether or not
// consecutive instructions share an accumulator.  The weight rows are therefore the M operand
// (blocks of 128 rows: a gate block and the matching up block, or two blocks of W_down) and the
// group's token rows are the N operand (a segment of up to 128 or 256 rows, rounded up to 16):
// the instruction time follows the number of tokens, so a group of 160 rows costs 160/256 of a
// full tile instead of two full instructions, and a handful of tokens cost the 48.5-cycle floor
// -- 8 KB of weights per 97 cycles, far more than HBM delivers per SM in that time.  The kernel
// stays bandwidth-bound from one token per expert up to the roofline ridge (Sec. 3.3: the
// layer's time is the time to load the activated experts), and full 256-token segments run the
// instruction at its full rate.  In TMEM a lane is a weight row (an output feature) and a
// column a token: an epilogue thread owns one feature and walks the tokens.
//
// Work partition.  Output features are independent, so the routed work is cut into (segment,
// tile, k chunk) items which the workers of the persistent grid claim at run time from a
// grid-wide counter: one that starts late or runs slowly takes less.
// The shared expert's rows are cut into (tile, k chunk, segment) units that are dealt
// round-robin to the CTAs; they depend on nothing the layer computes, so they run before the
// routing result exists.  Tiles have at most 128 features (gate/up: two blocks, gate and up)
// or 256 (down: two blocks).  The units of one shared tile run at the same time on
// neighbouring CTAs and meet in L2.
//
// Between the passes.  The gate/up pass counts, per segment, the 16-column units of h its
// epilogue warps have stored (a releasing reduction); the down pass starts while the gate/up
// pass is still running and fetches a segment's rows of h once the segment's count is
// complete (acquire load, then a proxy fence before the TMA loads).
//
// Two ring geometries, chosen by the host per call.  Streaming (segments of up to 128 rows): a
// weight slot holds two 64-element k boxes of one tile (64 KB for a full tile), so that one
// producer/consumer hand-shake moves enough bytes to keep HBM busy and every weight row is
// requested in 256 contiguous bytes; two sets of accumulators, so the epilogue of one tile
// runs under the instructions of the next.  Contraction (segments of up to 256 rows, for
// groups in the hundreds of rows): one k box per slot (32 KB) and per token entry, one set of
// accumulators of 2 x 256 columns.  The token operand lives in a second ring whose entries are
// sized by the segment's row count and never wrap.
//
// CTA pairs.  In the contraction geometry, and in the streaming one beyond 128 tokens
// (ffn_pairs), a cluster of two CTAs works on a tile of twice the features with tcgen05
// cta_group::2: each CTA loads its half of the weight rows and half of the token rows, the
// tensor cores of both read both halves of the tokens, and each CTA's TMEM and epilogue get its
// half of the features for all tokens.  What bounds the contraction is bytes: each SM is filled at
// no more than about 44 bytes per clock, a 256 x 256 tile of a single CTA wants 64 at the full
// instruction rate and 256 x 160 wants 81; a pair's CTA wants 47 and 66.  The leader (even CTA)
// claims the work for both, its barriers count the bytes of both and its commits release the slots
// of both.  Layer at the power cap, single CTAs -> pairs when this was taken up, medians of three
// runs of either in turn: Qwen2 shape T = 1280 1300 -> 1266 us, Mixtral shape T = 1280 1163 -> 1123.
//
// CTA = 11 warps.  warp 0: weight producer, warp 1: MMA issuer (idle in a pair's second CTA) and
// owner of the TMEM allocation, warp 2: token-operand producer (in all three the warp runs in
// step and one elected lane issues), warps 3..10: epilogue, two warps per TMEM lane quarter that
// take alternate 16-token chunks (tcgen05.ld, SwiGLU, transposition, 16-byte bf16 stores): where no
// second set of accumulators exists the epilogue is not hidden behind the next tile, and two warps
// per scheduler hide its latencies.  Rings and the accumulator sets are handed over through
// mbarriers.  Every wait is bounded: when one gives up it raises the CTA's abort flag and the device
// status word, all roles leave their loops (the other CTA of a pair by its own limits), TMEM is
// freed and the kernel returns.
//
// Programmatic dependent launch: the kernels may start while their predecessor in the stream
// is still running.  Work that depends only on the caller's inputs (shared-expert tiles in the
// gate/up pass, weight prefetch in the down pass) is done before griddepcontrol.wait, so it
// overlaps the routing kernels; everything produced inside the layer is touched after it,
// except h, which the down pass takes segment by segment as described above.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "tc_ptx.cuh"

#include "ffn_geometry.h"
#include "ffn_walk.cuh"

namespace moe {

// Tensor maps of one pass: weights [kind][matrix][box height], token operand [kind][box height].
struct FfnMaps {
    CUtensorMap w[2][2][FF_HEIGHTS];
    CUtensorMap x[2][FF_HEIGHTS];
};

// ---- kernel ----------------------------------------------------------------------------

// One output value of an epilogue thread: h = silu(g) * u (GATED) or the plain sum, as bf16.
template <bool GATED>
__device__ __forceinline__ __nv_bfloat16 epilogue_value(uint32_t g, uint32_t u)
{
    float v = __uint_as_float(g);
    if (GATED)
        v = silu_f(v) * __uint_as_float(u);
    return __float2bfloat16_rn(v);
}

// Epilogue transposition.  An epilogue thread owns one output feature (its TMEM lane) and
// holds that feature's values for 16 consecutive tokens, but the outputs are token-major
// (features contiguous).  Two-byte stores of single values cost a fifth of the whole pass at
// large token counts, so the warp first exchanges values with three rounds of shuffles
// (lane distances 1, 2, 4): afterwards every lane holds, for two of the 16 tokens, eight
// consecutive features as one 16-byte vector.
//   in:  w[c]  bf16 bits (low half) of this lane's feature for token c, c = 0..15
//   out: v[i]  features 8*(lane>>3) .. +7 of token  tok[i],  i = 0, 1
__device__ __forceinline__ void transpose_16x32(const uint32_t (&w)[16], int lane, uint4 (&v)[2],
                                                int (&tok)[2])
{
    const bool b1 = lane & 1, b2 = lane & 2, b4 = lane & 4;
    // distance 1: pairs of features; even lanes keep tokens 0-7, odd lanes tokens 8-15
    uint32_t p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t keep = b1 ? w[8 + i] : w[i];
        const uint32_t send = b1 ? w[i] : w[8 + i];
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, 1);
        p[i] = b1 ? (recv | (keep << 16)) : (keep | (recv << 16));
    }
    // distance 2: four features; the lane of the lower pair keeps the first four of its tokens
    uint32_t q0[4], q1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t keep = b2 ? p[4 + i] : p[i];
        const uint32_t send = b2 ? p[i] : p[4 + i];
        const uint32_t recv = __shfl_xor_sync(0xffffffffu, send, 2);
        q0[i] = b2 ? recv : keep;
        q1[i] = b2 ? keep : recv;
    }
    // distance 4: eight features, two tokens
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t k0 = b4 ? q0[2 + i] : q0[i], k1 = b4 ? q1[2 + i] : q1[i];
        const uint32_t s0 = b4 ? q0[i] : q0[2 + i], s1 = b4 ? q1[i] : q1[2 + i];
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, s0, 4);
        const uint32_t r1 = __shfl_xor_sync(0xffffffffu, s1, 4);
        v[i] = b4 ? make_uint4(r0, r1, k0, k1) : make_uint4(k0, k1, r0, r1);
        tok[i] = (b1 ? 8 : 0) + (b2 ? 4 : 0) + (b4 ? 2 : 0) + i;
    }
}

// GATED: W_gate and W_up tiles -> h = silu(g) * u.   !GATED: W_down tiles -> y.
template <bool GATED, bool PAIR>
__global__ void __launch_bounds__(FF_THREADS, 1)
ffn_fused_kernel(const FfnArgs args, const __grid_constant__ FfnMaps maps)
{
    constexpr int NW = GATED ? 2 : 1;  // weight matrices per tile (gate and up: one block each)

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * FF_STEPS + 4 + 2 * FF_CLAIMS];
    __shared__ uint32_t tmem_base_holder;
    __shared__ int abort_flag[2];  // [0] raised by the first wait that gives up, [1] wait limit (us)
    __shared__ __align__(16) int claim_data[FF_CLAIMS * FF_CLAIM_WORDS];

    const int NS = args.n_w_slots;
    // (only pairs run the contraction geometry)
    const int kb = PAIR ? args.kboxes : 2;
    // TMEM: a set of accumulators is two blocks (gate and up, or two blocks of 128 down rows) of
    // acc_block columns each; two sets of 2 x 128 columns, or one set of 2 x 256
    const int acc_sets = PAIR ? args.acc_sets : 2;
    const uint32_t acc_block = acc_sets == 2 ? 128u : 256u;
    // token ring first (an MMA reads exactly the rows of its entry, rounded up to 16; a weight
    // block is read as 128 rows, which for a shorter tile ends inside the slot's capacity)
    const uint32_t ring_x = (smem_u32(smem_raw) + 1023u) & ~1023u;  // swizzle needs 1 KB alignment
    const uint32_t ring_w = ring_x + (uint32_t)args.x_units * FF_X_UNIT;
    const uint32_t bar0 = smem_u32(bars);
    // One barrier pair per k step in flight (a weight slot and a token entry, consumed together),
    // step j on pair j % FF_STEPS.  full: both producers' bytes; empty: the step's instructions
    // have read them.  The weight producer refills slot j % NS once step j - NS is consumed.
    auto full = [&](int j) { return bar0 + 8u * (j % FF_STEPS); };
    auto empty = [&](int j) { return bar0 + 8u * (FF_STEPS + j % FF_STEPS); };
    auto parity = [](int j) { return (uint32_t)(j / FF_STEPS) & 1u; };
    auto acc_full = [&](int b) { return bar0 + 8u * (2 * FF_STEPS + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (2 * FF_STEPS + 2 + b); };
    const uint32_t claim_full0 = bar0 + 8u * (2 * FF_STEPS + 4);
    const uint32_t claim_empty0 = claim_full0 + 8u * FF_CLAIMS;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // pair: the leader's barriers count the bytes that land in both CTAs, its issuer feeds both
    // tensor pipes and releases the slots of both
    const int rank = PAIR ? (int)(blockIdx.x & 1) : 0;
    constexpr int CTAS = PAIR ? 2 : 1;
    auto leader_bar = [&](uint32_t bar) { return PAIR ? map_to_rank(bar, 0) : bar; };

    if (threadIdx.x == 0) {
        abort_flag[0] = 0;
        abort_flag[1] = args.wait_us;
        for (int j = 0; j < FF_STEPS; ++j) {
            mbar_init(full(j), 2);
            mbar_init(empty(j), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full(b), 1);
            mbar_init(acc_empty(b), CTAS * FF_EPI_WARPS);
        }
        for (int i = 0; i < FF_CLAIMS; ++i) {
            mbar_init(claim_full0 + 8u * i, 1);
            mbar_init(claim_empty0 + 8u * i, CTAS * FF_CLAIM_READERS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base_holder)),
                         "r"(FF_TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tmem_base_holder)),
                         "r"(FF_TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR)
        cluster_barrier();  // the other CTA's barriers are initialised, its TMEM is allocated
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_holder;
    volatile int *abortp = abort_flag;
    const ClaimRing claims{claim_data, claim_full0, claim_empty0, abortp, args.status,
                           PAIR ? map_to_rank(smem_u32(claim_data), rank ^ 1) : 0u,
                           PAIR ? map_to_rank(claim_full0, rank ^ 1) : 0u, leader_bar(claim_empty0)};

    if (warp == 0) {
        // ---------------- weight producer ----------------
        // As in the issuer, all lanes in step with uniform values and one elected lane issues the
        // copies.  With the loop in one lane's branch the issue of a copy cost several hundred
        // cycles: tiles of 32 rows, whose passes that bounds, took 361 us at T = 77 on the Qwen1.5
        // shape against 303; with the tiles in use 182 -> 180, T = 32 162 -> 158, the Qwen2 shape
        // with skewed routing at T = 320 778 -> 760 (one barrier per k step included).
        //
        // gate/up pass: the shared expert's weights and x are the caller's inputs, so those
        // items run before the wait.  Down pass: every weight tile may be fetched ahead --
        // the launch order guarantees that the plan is complete when this kernel starts.
        ItemWalk<PAIR> walk(args, claims, rank == 0, !GATED);
        const uint64_t pol_once = l2_policy_evict_first();
        bool launched = !GATED;
        if (!GATED)
            griddep_launch();
        int slot = 0, step = 0;
        bool ok = true;
        Item it;
        while (ok && walk.next(it)) {
            if (!launched && walk.synced) {
                griddep_launch();  // after the wait: dependents may rely on the plan
                launched = true;
            }
            const int grp = warp_uniform(it.grp), w_once = warp_uniform(it.w_once);
            const int hc = warp_uniform(it.h) / CTAS;  // this CTA's rows of the tile
            const uint32_t tile_bytes = (uint32_t)hc * 128u;
            // expert = 0 for the shared kind
            const int wrow = warp_uniform(it.expert * args.rows[0] + it.f0) + rank * hc;
            const int k_begin = warp_uniform(it.k0), k_end = warp_uniform(it.k1);
            for (int k0 = k_begin; k0 < k_end; k0 += 64 * kb) {
                const int nbox = min(kb, (k_end - k0 + 63) >> 6);
                const bool free = step < NS || mbar_wait(empty(step - NS), parity(step - NS), abortp, args.status);
                if (!__all_sync(0xffffffffu, free)) {
                    ok = false;
                    break;
                }
                const uint32_t base = ring_w + slot * args.w_slot_bytes;
                const uint32_t bar = leader_bar(full(step));
                if (elect_one()) {
                    if (rank == 0)
                        mbar_expect_tx(full(step), CTAS * nbox * NW * tile_bytes);
                    for (int b = 0; b < nbox; ++b) {
#pragma unroll
                        for (int m = 0; m < NW; ++m) {
                            // the tile as boxes of 128, 64, 32 and 16 rows, stacked
                            uint32_t dst = base + (uint32_t)(b * NW + m) * tile_bytes;
                            int row = wrow, rem = hc;
                            while (rem > 0) {
                                const int hi = rem >= 128 ? 0 : (rem >= 64 ? 1 : (rem >= 32 ? 2 : 3));
                                const int bh = 128 >> hi;
                                const CUtensorMap *map = &maps.w[grp][m][hi];
                                if (PAIR && w_once)
                                    tma_load_2d_pair_hint(dst, map, bar, k0 + 64 * b, row, pol_once);
                                else if (PAIR)
                                    tma_load_2d_pair(dst, map, bar, k0 + 64 * b, row);
                                else if (w_once)
                                    tma_load_2d_hint(dst, map, bar, k0 + 64 * b, row, pol_once);
                                else
                                    tma_load_2d(dst, map, bar, k0 + 64 * b, row);
                                dst += (uint32_t)bh * 128u;
                                row += bh;
                                rem -= bh;
                            }
                        }
                    }
                }
                __syncwarp();
                ++step;
                if (++slot == NS)
                    slot = 0;
            }
        }
        if (!walk.synced)
            walk.sync(true);
        if (!launched)
            griddep_launch();
    } else if (warp == 2) {
        // ---------------- token-operand producer ----------------
        // down pass: h is written by the preceding kernel, which may still be running; a
        // segment's rows are fetched once its progress counter says they are complete
        ItemWalk<PAIR> walk(args, claims, false, !GATED);
        TokenRing ring(args.x_units);
        int starts[FF_STEPS];
        int seen = -1;  // (group kind, segment) key last found complete
        const uint64_t pol_keep = l2_policy_evict_last();
        bool ok = true;
        Item it;
        while (ok && walk.next(it)) {
            const int grp = warp_uniform(it.grp);
            if (!GATED) {
                const int key = (it.grp << 30) | it.seg;
                if (key != seen) {
                    // every epilogue warp of the gate/up pass counts the 16-column units
                    // of h it has finished for the segment
                    const bool done = counter_wait(args.done[it.grp] + it.seg,
                                                   (args.K[it.grp] >> 4) * FF_EPI_WARPS, abortp, args.status);
                    seen = key;
                    ok = __all_sync(0xffffffffu, done);
                    if (!ok)
                        break;
                    // rows written through the generic proxy, read below by the async proxy
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                }
            }
            const int pieces = token_pieces<PAIR>(warp_uniform(it.n));  // this CTA's share of the rows
            const int m = pieces * kb;
            const int xrow = warp_uniform(it.row0) + rank * (pieces << 4);
            const int k_begin = warp_uniform(it.k0), k_end = warp_uniform(it.k1);
            for (int k0 = k_begin; k0 < k_end; k0 += 64 * kb) {
                const int nbox = min(kb, (k_end - k0 + 63) >> 6);
                const int j = ring.count;
                const int at = ring.place(m);
                while (ok && ring.must_release()) {
                    const bool free = mbar_wait(empty(ring.released), parity(ring.released), abortp, args.status);
                    ok = __all_sync(0xffffffffu, free);
                    ring.release(starts);
                }
                if (!ok)
                    break;
                ring.issued(starts);
                const uint32_t base = ring_x + (uint32_t)at * FF_X_UNIT;
                const uint32_t bar = leader_bar(full(j));
                if (elect_one()) {
                    if (rank == 0)
                        mbar_expect_tx(full(j), (uint32_t)(CTAS * nbox * pieces) * FF_X_UNIT);
                    for (int b = 0; b < nbox; ++b) {
                        // the entry's rows as boxes of 128, 64, 32 and 16 rows
                        uint32_t dst = base + (uint32_t)(b * pieces) * FF_X_UNIT;
                        int row = xrow, rem = pieces << 4;
                        while (rem > 0) {
                            const int hi = rem >= 128 ? 0 : (rem >= 64 ? 1 : (rem >= 32 ? 2 : 3));
                            const int bh = 128 >> hi;
                            if (PAIR)
                                tma_load_2d_pair_hint(dst, &maps.x[grp][hi], bar, k0 + 64 * b, row, pol_keep);
                            else
                                tma_load_2d_hint(dst, &maps.x[grp][hi], bar, k0 + 64 * b, row, pol_keep);
                            dst += (uint32_t)bh * 128u;
                            row += bh;
                            rem -= bh;
                        }
                    }
                }
                __syncwarp();
            }
        }
        if (PAIR)  // the leader's last releases have arrived before this CTA may exit
            for (; ok && ring.released < ring.count; ++ring.released)
                ok = __all_sync(0xffffffffu, mbar_wait(empty(ring.released), parity(ring.released), abortp,
                                                       args.status));
        if (!walk.synced)
            walk.sync(true);
        if (!GATED)
            griddep_wait();  // no kernel of the chain completes before its predecessor
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // All lanes walk, wait and compute, and the values of an item that came through shared
        // memory are made warp-uniform for the compiler; one elected lane issues.  With the whole
        // loop in one lane's branch the operands of every instruction had to be moved to the
        // uniform registers the tensor pipe reads, and the issue bounded the pass: about 140
        // cycles per instruction where N / 2 = 80 to 128 are its time (Qwen2 shape, T = 1280).
        // Layer, before -> after: Qwen1.5 shape T = 5 77.4 -> 71.0 us, T = 640 270 -> 258,
        // Mixtral shape T = 1280 1256 -> 1218, DeepSeek-V3 shape T = 128 3261 -> 3178.
        if (rank == 0) {
            ItemWalk<PAIR> walk(args, claims, false, !GATED);
            XRingWalk ring(args.x_units);
            int sw = 0;
            bool ok = true;
            int n_items = 0;
            Item it;
            while (ok && walk.next(it)) {
                // the accumulator set is waited for right before the item's first instruction, so
                // that its operands are already being fetched while the epilogue drains the set
                const int set = n_items % acc_sets;
                const uint32_t acc_par = ((uint32_t)(n_items / acc_sets) & 1u) ^ 1u;
                ++n_items;
                const uint32_t d0 = tmem_base + (uint32_t)set * 2u * acc_block;
                const int hc = warp_uniform(it.h) / CTAS;
                const uint32_t tile_bytes = (uint32_t)hc * 128u;
                const int pieces = token_pieces<PAIR>(warp_uniform(it.n));
                // M = 128 per CTA, N = token rows
                const uint32_t idesc = umma_idesc_bf16(CTAS * (pieces << 4), CTAS * 128);
                // weight blocks of the tile: gate and up, or the 128-row halves of a down tile
                const int nblk = GATED ? 2 : (hc + 127) >> 7;
                // descriptor steps in 16-byte units: to the next block, to the next k box
                const uint32_t blk16 = (GATED ? tile_bytes : 128u * 128u) >> 4;
                const uint64_t w_box16 = (uint64_t)((NW * tile_bytes) >> 4);
                const uint64_t x_box16 = (uint64_t)((pieces * FF_X_UNIT) >> 4);
                const int n_box = warp_uniform((it.k1 - it.k0 + 63) >> 6);  // k boxes of the item
                uint32_t accum = 0;
                for (int box = 0; box < n_box; box += kb) {
                    const int nbox = min(kb, n_box - box);
                    const int j = ring.count;
                    const int at = ring.place(pieces * kb);
                    const uint32_t xbase = ring_x + (uint32_t)at * FF_X_UNIT;
                    bool ready = mbar_wait(full(j), parity(j), abortp, args.status);
                    if (box == 0)
                        ready = ready && mbar_wait<PAIR>(acc_empty(set), acc_par, abortp, args.status);
                    if (!__all_sync(0xffffffffu, ready)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    uint64_t w_desc = umma_desc_sw128(ring_w + sw * args.w_slot_bytes);
                    uint64_t x_desc = umma_desc_sw128(xbase);
                    if (elect_one()) {
                        for (int b = 0; b < nbox; ++b) {
                            if (nblk == 2)
                                issue_k_box<2, PAIR>(d0, acc_block, w_desc, blk16, x_desc, idesc, accum);
                            else
                                issue_k_box<1, PAIR>(d0, acc_block, w_desc, blk16, x_desc, idesc, accum);
                            w_desc += w_box16;
                            x_desc += x_box16;
                            accum = 1u;
                        }
                        umma_commit<PAIR>(empty(j));  // reusable once these MMAs have read them
                        if (box + kb >= n_box)
                            umma_commit<PAIR>(acc_full(set));  // accumulators complete
                    }
                    __syncwarp();
                    accum = 1u;
                    if (++sw == NS)
                        sw = 0;
                }
            }
            if (!walk.synced)
                walk.sync(true);
        }
    } else {
        // ---------------- epilogue (warps 3..10) ----------------
        // down pass: its outputs are read by nothing older than this call's combine, so the
        // stores need not wait for the preceding kernel (the token producer does, per segment)
        const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31 belong to this warp
        const int chunk0 = warp >= 7 ? 16 : 0;  // the quarter's second warp takes the odd chunks
        ItemWalk<PAIR> walk(args, claims, false, !GATED);
        int n_items = 0;
        Item it;
        for (;;) {
            // the walk is identical in all lanes; griddepcontrol.wait inside next() is
            // executed by every lane
            if (!walk.next(it))
                break;
            const int set = n_items % acc_sets;
            const uint32_t acc_phase = (uint32_t)(n_items / acc_sets) & 1u;
            ++n_items;
            // every lane waits; the vote makes the decision uniform and reconverges the warp
            // for the warp-collective tcgen05.ld below
            const bool ready = mbar_wait(acc_full(set), acc_phase, abortp, args.status);
            if (!__all_sync(0xffffffffu, ready))
                break;
            tc_fence_after();
            // a thread owns one weight row (output feature) of a block and walks the tokens
            const int hc = it.h / CTAS;
            const int nblk = GATED ? 1 : (hc + 127) >> 7;  // gate and up are read together
            const int ld = args.out_ld[it.grp];
            const int npad = pieces16(it.n) << 4;
            for (int m = 0; m < nblk; ++m) {
                const int rows_blk = GATED ? hc : min(128, hc - 128 * m);
                if (quarter * 32 >= rows_blk)
                    break;  // this warp's lanes lie beyond the tile (uniform)
                // after the transposition this lane stores features 8 * (lane >> 3) .. + 7 of
                // the warp's 32 (tiles are multiples of 16 features: all eight exist or none)
                const int fgrp = quarter * 32 + 8 * (lane >> 3);
                const bool grp_ok = fgrp < rows_blk;
                __nv_bfloat16 *out = args.out[it.grp] + it.out_off + (size_t)it.row0 * ld + it.f0 +
                                     rank * hc + 128 * m + fgrp;
                const uint32_t t0 = tmem_base + ((uint32_t)(quarter * 32) << 16) +
                                    (uint32_t)set * 2u * acc_block + (uint32_t)m * acc_block;
                // two register buffers: the TMEM load of this warp's next 16 tokens is in flight
                // while the current 16 are converted, transposed and stored
                uint32_t g[2][16], u[2][16];
                if (chunk0 < npad) {
                    tmem_ld16(t0 + chunk0, g[0]);
                    if (GATED)
                        tmem_ld16(t0 + acc_block + chunk0, u[0]);
                }
#pragma unroll 1
                for (int c = chunk0; c < npad; c += 64) {
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int cc = c + 32 * half;
                        if (cc < npad) {
                            tmem_ld_wait();
                            if (cc + 32 < npad) {
                                tmem_ld16(t0 + cc + 32, g[half ^ 1]);
                                if (GATED)
                                    tmem_ld16(t0 + acc_block + cc + 32, u[half ^ 1]);
                            }
                            if (!GATED && args.f32_out) {
                                // a lane's values as they are: 128 contiguous bytes per token
                                float *of = reinterpret_cast<float *>(args.out[it.grp]) + it.out_off +
                                            (size_t)(it.row0 + cc) * ld + it.f0 + rank * hc + 128 * m +
                                            quarter * 32 + lane;
                                if (quarter * 32 + lane < rows_blk) {
#pragma unroll
                                    for (int i = 0; i < 16; ++i)
                                        if (cc + i < it.n)
                                            of[(size_t)i * ld] = __uint_as_float(g[half][i]);
                                }
                                continue;
                            }
                            uint32_t w[16];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const __nv_bfloat16 val = epilogue_value<GATED>(g[half][i], u[half][i]);
                                w[i] = (uint32_t)__bfloat16_as_ushort(val);
                            }
                            uint4 v[2];
                            int tok[2];
                            transpose_16x32(w, lane, v, tok);
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                if (grp_ok && cc + tok[i] < it.n)
                                    *reinterpret_cast<uint4 *>(out + (size_t)(cc + tok[i]) * ld) = v[i];
                        }
                    }
                }
            }
            tc_fence_before();
            if (GATED)  // the down pass fetches these rows with TMA (async proxy)
                asm volatile("fence.proxy.async.global;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                if (PAIR)
                    mbar_arrive_cluster(leader_bar(acc_empty(set)));
                else
                    mbar_arrive(acc_empty(set));
                if (GATED) {
                    // publish: this warp's part of the tile is in h (a releasing reduction: the
                    // warp does not wait for its stores to become visible, the counter does)
                    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(args.done[it.grp] + it.seg),
                                 "r"(hc >> 4)
                                 : "memory");
                }
            }
        }
        if (!walk.synced)
            walk.sync(true);
    }

    if (*abortp) {
        // A wait gave up.  Copies and tensor-core instructions already issued may still be in
        // flight: every thread that sees the flag (the one that raised it always does) holds
        // the CTA for a millisecond, far longer than any of them takes, before shared memory
        // and TMEM are given back.
        const uint64_t t0 = global_ns();
        while (global_ns() - t0 < 1000000ull) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR)
        cluster_barrier();  // nothing of the other CTA refers to this one's memory any more
    if (warp == 1) {
        __syncwarp();  // the deallocation is warp-collective
        tc_fence_after();
        if (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                         "r"(FF_TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                         "r"(FF_TMEM_COLS)
                         : "memory");
    }
}

// ---- self-test of the bounded wait ---------------------------------------------------------

// Waits, with the given limit, for a progress counter that nothing advances: the wait the down
// pass uses for the gate/up pass's counters must give up, raise the status word and return.
__global__ void wait_limit_selftest_kernel(int32_t *status, int32_t *never_set, int limit_us)
{
    __shared__ int abort_flag[2];
    if (threadIdx.x == 0) {
        abort_flag[0] = 0;
        abort_flag[1] = limit_us;
        status[0] = 0;
        status[1] = STATUS_MAGIC;
        never_set[0] = 0;
        __threadfence();
        counter_wait(never_set, 1, abort_flag, status);
    }
}

cudaError_t launch_wait_limit_selftest(int32_t *status, int32_t *never_set, int limit_us,
                                       cudaStream_t s)
{
    wait_limit_selftest_kernel<<<1, 32, 0, s>>>(status, never_set, limit_us);
    return cudaGetLastError();
}

// ---- gather of the token rows into sorted order (B operand of the gate/up pass) ---------

constexpr int GATHER_UNROLL = 8;

// One warp per sorted row: the source token is looked up once per row (all lanes read the same
// word), then the row is copied in passes of GATHER_UNROLL x 512 bytes whose loads are all in
// flight before the first store.
__global__ void __launch_bounds__(256)
gather_rows_kernel(const __nv_bfloat16 *__restrict__ x, const int32_t *__restrict__ perm, int A,
                   int H, int top_k, __nv_bfloat16 *__restrict__ x_sorted)
{
    griddep_launch();
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    const int vec_per_row = H >> 3;
    for (int r = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); r < A; r += warps) {
        const int t = perm[r] / top_k;
        const uint4 *src = reinterpret_cast<const uint4 *>(x + (size_t)t * H);
        uint4 *dst = reinterpret_cast<uint4 *>(x_sorted + (size_t)r * H);
        for (int v0 = lane; v0 < vec_per_row; v0 += 32 * GATHER_UNROLL) {
            uint4 d[GATHER_UNROLL];
#pragma unroll
            for (int u = 0; u < GATHER_UNROLL; ++u)
                if (v0 + 32 * u < vec_per_row)
                    d[u] = src[v0 + 32 * u];
#pragma unroll
            for (int u = 0; u < GATHER_UNROLL; ++u)
                if (v0 + 32 * u < vec_per_row)
                    dst[v0 + 32 * u] = d[u];
        }
    }
}

// The same from the token's side, where the inverse permutation is at hand (a layer call): a warp
// reads a piece of 2048 columns once and writes it to its top_k places.  Bound by the writes;
// gather_rows_kernel also reads every row top_k times.  Alone, us: DeepSeek-V3 shape T = 3072 96 -> 71
// (5.6 TB/s of rows read and written once), T = 1536 43.5 -> 35.7, Qwen2 T = 1280 and 2048 equal;
// layer, 64 experts top-8 of 256, T = 2048: hidden 256 63.1 -> 56.7, 1024 114.1 -> 111.3.
__global__ void __launch_bounds__(256)
gather_tokens_kernel(const __nv_bfloat16 *__restrict__ x, const int32_t *__restrict__ inv_perm, int T,
                     int H, int top_k, __nv_bfloat16 *__restrict__ x_sorted)
{
    griddep_launch();
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    const int vec_per_row = H >> 3;
    const int pieces = (vec_per_row + 32 * GATHER_UNROLL - 1) / (32 * GATHER_UNROLL);
    for (int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); i < T * pieces; i += warps) {
        const int t = i / pieces, v0 = (i - t * pieces) * 32 * GATHER_UNROLL + lane;
        const int place = lane < top_k ? inv_perm[(size_t)t * top_k + lane] : 0;
        const uint4 *src = reinterpret_cast<const uint4 *>(x + (size_t)t * H);
        uint4 d[GATHER_UNROLL];
#pragma unroll
        for (int u = 0; u < GATHER_UNROLL; ++u)
            if (v0 + 32 * u < vec_per_row)
                d[u] = src[v0 + 32 * u];
        for (int j = 0; j < top_k; ++j) {
            const int row = __shfl_sync(0xffffffffu, place, j);
            uint4 *dst = reinterpret_cast<uint4 *>(x_sorted + (size_t)row * H);
#pragma unroll
            for (int u = 0; u < GATHER_UNROLL; ++u)
                if (v0 + 32 * u < vec_per_row)
                    dst[v0 + 32 * u] = d[u];
        }
    }
}

cudaError_t launch_gather_tokens(const moe_config_t &c, const __nv_bfloat16 *x, const int32_t *inv_perm,
                                 int T, __nv_bfloat16 *x_sorted, cudaStream_t s)
{
    const int vec = c.hidden >> 3, pieces = (vec + 32 * GATHER_UNROLL - 1) / (32 * GATHER_UNROLL);
    size_t blocks = ((size_t)T * pieces + 7) / 8;  // a piece of a row per warp, eight warps per CTA
    const size_t cap = (size_t)sm_count() * gather_ctas_per_sm(c, T, c.shared_inter > 0);
    if (blocks > cap)
        blocks = cap;
    return launch_pdl(gather_tokens_kernel, dim3((unsigned)blocks), dim3(256), 0, s, x, inv_perm, T,
                      c.hidden, c.top_k, x_sorted);
}

cudaError_t launch_gather_rows(const moe_config_t &c, const __nv_bfloat16 *x, const int32_t *perm,
                               int T, __nv_bfloat16 *x_sorted, cudaStream_t s)
{
    const int A = T * c.top_k;
    size_t blocks = ((size_t)A + 7) / 8;  // a row per warp, eight warps per CTA
    const size_t cap = (size_t)sm_count() * gather_ctas_per_sm(c, T, true);
    if (blocks > cap)
        blocks = cap;
    return launch_pdl(gather_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, s, x, perm, A,
                      c.hidden, c.top_k, x_sorted);
}

// ---- host side: geometry, tensor maps and launches ---------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// 2-D bf16 tensor [rows, cols] (cols contiguous), box = 64 columns x box_rows, 128-byte swizzle.
bool make_tma_map_2d_bf16(CUtensorMap *m, const void *base, uint64_t rows, uint64_t cols,
                          uint32_t box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn)
        return false;
    if (base == nullptr || rows == 0 || cols == 0) {
        memset(m, 0, sizeof *m);  // group kind not present: never used by the kernel
        return true;
    }
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 2};
    const cuuint32_t box[2] = {64, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// the four box heights of one matrix
static bool make_weight_maps(CUtensorMap (&m)[FF_HEIGHTS], const void *base, uint64_t rows, uint64_t cols)
{
    for (int i = 0; i < FF_HEIGHTS; ++i)
        if (!make_tma_map_2d_bf16(&m[i], base, rows, cols, 128u >> i))
            return false;
    return true;
}

// Encoded tensor maps of recent launches.  A serving loop calls the layer with the same
// weights, workspace and token count again and again; encoding the twenty maps of a pass costs
// more host time than the launch itself, so the maps are kept, keyed by everything that enters
// them (device, pass, base pointers, extents).  A few dozen entries, replaced in turn.
struct MapKey {
    int device, gated;
    const void *ptr[7];
    uint64_t dim[6];
};
struct MapCacheEntry {
    bool used;
    MapKey key;
    FfnMaps maps;
};
constexpr int FF_MAP_CACHE = 48;
static MapCacheEntry g_map_cache[FF_MAP_CACHE];
static int g_map_cache_next = 0, g_map_cache_last = 0;
static std::mutex g_map_cache_mutex;

static bool map_cache_lookup(const MapKey &key, FfnMaps &out)
{
    std::lock_guard<std::mutex> lock(g_map_cache_mutex);
    for (int n = 0; n < FF_MAP_CACHE; ++n) {
        const int i = (g_map_cache_last + n) % FF_MAP_CACHE;  // the last hit first
        if (g_map_cache[i].used && memcmp(&g_map_cache[i].key, &key, sizeof key) == 0) {
            out = g_map_cache[i].maps;
            g_map_cache_last = i;
            return true;
        }
    }
    return false;
}

static void map_cache_store(const MapKey &key, const FfnMaps &maps)
{
    std::lock_guard<std::mutex> lock(g_map_cache_mutex);
    MapCacheEntry &e = g_map_cache[g_map_cache_next];
    e.used = true;
    e.key = key;
    e.maps = maps;
    g_map_cache_last = g_map_cache_next;
    g_map_cache_next = (g_map_cache_next + 1) % FF_MAP_CACHE;
}

static MapKey map_key(bool gated, const void *p0, const void *p1, const void *p2, const void *p3,
                      const void *p4, const void *p5, const void *p6, uint64_t d0, uint64_t d1,
                      uint64_t d2, uint64_t d3, uint64_t d4, uint64_t d5)
{
    MapKey k;
    memset(&k, 0, sizeof k);  // padding bytes take part in the comparison
    cudaGetDevice(&k.device);
    k.gated = gated ? 1 : 0;
    const void *p[7] = {p0, p1, p2, p3, p4, p5, p6};
    const uint64_t d[6] = {d0, d1, d2, d3, d4, d5};
    memcpy(k.ptr, p, sizeof p);
    memcpy(k.dim, d, sizeof d);
    return k;
}

int geometry_override()
{
    static const int v = [] {
        const char *e = getenv("MOE_FF_WIDE");
        return !e ? -1 : (e[0] == '1' ? 1 : (e[0] == '0' ? 0 : -1));
    }();
    return v;
}

bool pairs_forced()
{
    static const bool v = [] {
        const char *e = getenv("MOE_FF_PAIR");
        return e && e[0] == '1';
    }();
    return v;
}

int ffn_segment_rows(const moe_config_t &c, int T) { return segment_rows(c, T); }

// Number of tiles the shared expert's rows are cut into.  The shared expert's work units are
// (tile, k chunk, segment); a unit should cost about the expected per-CTA share of the whole
// pass (or less), with the tile height within [min_tile, max_tile] rows (a weight block
// costs the same instruction time whether it holds 16 rows or 128).
static int shared_tile_count(const moe_config_t &c, int T, int rows_routed, int rows_shared,
                             int K_routed, int K_shared, int ksplit, int min_tile, int max_tile)
{
    const FfnWorkers wk = ffn_workers(c, T);
    const int unit = 16 * wk.ctas;  // (a pair's tiles: twice the height, units of 32 rows)
    const int seg_s = shared_segment_rows(c, T), seg_r = segment_rows(c, T);
    const int nseg_s = (T + seg_s - 1) / seg_s;
    const int units = rows_shared / unit;
    const double k_ratio = (double)K_shared / K_routed;  // cost of a shared row unit per segment
    const double n_act = expected_active_experts(c.n_experts, c.top_k, T);
    const double segs_r = n_act * ceil((double)T * c.top_k / n_act / seg_r);
    const double total = units * k_ratio * nseg_s + segs_r * (rows_routed / unit);
    int tu = (int)ceil(total / wk.count / (k_ratio / ksplit));
    if (tu < (min_tile >> 4))
        tu = min_tile >> 4;
    if (tu > (max_tile >> 4))
        tu = max_tile >> 4;
    return (units + tu - 1) / tu;
}

template <bool GATED, bool PAIR>
static cudaError_t launch_ffn(FfnArgs &a, const FfnMaps &maps, cudaStream_t s)
{
    // the opt-in to large dynamic shared memory is a per-device attribute of the kernel
    static DeviceOnce configured;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess)
        return cudaErrorInvalidDevice;
    if (!configured.done(dev)) {
        cudaError_t e = cudaFuncSetAttribute(ffn_fused_kernel<GATED, PAIR>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             FF_SMEM_LIMIT - 512);
        if (e != cudaSuccess)
            return e;
        configured.mark(dev);
    }
    const size_t smem = (size_t)a.x_units * FF_X_UNIT + (size_t)a.n_w_slots * a.w_slot_bytes + 1024;
    if (a.n_w_slots < 2 || smem > FF_SMEM_LIMIT - 512 || (!PAIR && a.seg_rows != FF_SEG))
        return cudaErrorInvalidConfiguration;
    const int grid = PAIR ? ffn_grid() & ~1 : ffn_grid();
    return launch_pdl<PAIR ? 2 : 1>(ffn_fused_kernel<GATED, PAIR>, dim3(grid), dim3(FF_THREADS), smem, s, a,
                                    maps);
}

cudaError_t launch_ffn_gateup(const moe_config_t &c, const moe_weights_t &w, const __nv_bfloat16 *x,
                              const __nv_bfloat16 *x_sorted, int T, PlanView plan, bool with_shared,
                              int routed_parts, __nv_bfloat16 *h, __nv_bfloat16 *h_shared,
                              int32_t *status, cudaStream_t s)
{
    const uint64_t A = (uint64_t)T * c.top_k, H = c.hidden, E = c.n_experts;
    FfnArgs a{};
    a.rows[0] = c.inter;
    a.rows[1] = c.shared_inter;
    a.K[0] = a.K[1] = c.hidden;
    a.max_tile = routed_tile_rows(c, T, routed_parts).up;
    a.shared_ksplit = 1;
    a.shared_kchunk = (c.hidden + 127) / 128 * 128;
    a.shared_tiles = with_shared ? shared_tile_count(c, T, c.inter, c.shared_inter, c.hidden, c.hidden,
                                                     1, 64, 128)
                                 : 0;
    ffn_geometry(c, T, a);
    a.wait_us = (int)(FF_WAIT_NS / 1000ull);
    FfnMaps maps;
    const MapKey key = map_key(true, w.w_gate, w.w_up, x_sorted, with_shared ? w.ws_gate : nullptr,
                               with_shared ? w.ws_up : nullptr, with_shared ? x : nullptr, nullptr, E,
                               (uint64_t)c.inter, H, A, with_shared ? (uint64_t)c.shared_inter : 0,
                               (uint64_t)T);
    if (!map_cache_lookup(key, maps)) {
        memset(&maps, 0, sizeof maps);
        bool ok = make_weight_maps(maps.w[0][0], w.w_gate, E * c.inter, H) &&
                  make_weight_maps(maps.w[0][1], w.w_up, E * c.inter, H) &&
                  make_weight_maps(maps.x[0], x_sorted, A, H);
        if (with_shared)
            ok = ok && make_weight_maps(maps.w[1][0], w.ws_gate, c.shared_inter, H) &&
                 make_weight_maps(maps.w[1][1], w.ws_up, c.shared_inter, H) &&
                 make_weight_maps(maps.x[1], x, T, H);
        if (!ok)
            return cudaErrorInvalidValue;
        map_cache_store(key, maps);
    }
    a.out[0] = h;
    a.out[1] = h_shared;
    a.out_ld[0] = c.inter;
    a.out_ld[1] = c.shared_inter;
    a.plan_header = plan.header;
    a.seg = plan.seg;
    a.max_seg = max_segments(c.n_experts, T * c.top_k);
    a.first_fixed = 1;
    a.claim_counter = plan.header + 2;
    a.done[0] = plan.done_routed;
    a.done[1] = plan.done_shared;
    a.routed_ksplit = 1;
    a.routed_kchunk = c.hidden;
    a.status = status;
    a.T = T;
    a.with_shared = with_shared ? 1 : 0;
    return ffn_pairs(c, T) ? launch_ffn<true, true>(a, maps, s) : launch_ffn<true, false>(a, maps, s);
}

// Length of a k chunk when K is cut into about `parts` pieces (a multiple of the 128-column
// weight slot), and the number of non-empty chunks that length gives.
static int split_chunk(int K, int parts) { return ((K + parts - 1) / parts + 127) / 128 * 128; }
static int split_parts(int K, int parts) { return (K + split_chunk(K, parts) - 1) / split_chunk(K, parts); }

// Expected number of (segment, tile) items of the routed down pass (counted with the wide
// segments, so that it never decreases with T).
static double routed_down_items(const moe_config_t &c, int T)
{
    const double n_act = expected_active_experts(c.n_experts, c.top_k, T);
    const double rows_per_group = (double)T * c.top_k / n_act;
    return ceil(n_act) * ceil(rows_per_group / FF_SEG_WIDE) * ((c.hidden + 255) / 256);
}

// k chunks of the routed groups' down projection.  While the pass has fewer than about three
// (segment, tile) items per CTA -- few tokens, or few experts with long reductions -- some SMs
// have no weight stream to pull and one SM cannot pull a tile faster than a fraction of what
// HBM delivers, so the reduction is cut; each chunk writes its own plane of y and the combine
// adds the planes.
int routed_down_parts(const moe_config_t &c, int T)
{
    int parts = (int)ceil(3.0 * ffn_grid() / routed_down_items(c, T));
    const int cap = c.inter / 1024;  // chunks below half a megabyte cost more than they level
    if (parts > cap)
        parts = cap;
    if (parts > ROUTED_SPLIT_MAX_PARTS)
        parts = ROUTED_SPLIT_MAX_PARTS;
    return parts < 1 ? 1 : split_parts(c.inter, parts);
}

size_t routed_split_max_rows(const moe_config_t &c, int T)
{
    if (c.inter / 1024 < 2)
        return 0;
    // largest T' <= T whose item count still asks for more than one part
    auto split = [&](int t) { return routed_down_items(c, t) < 3.0 * ffn_grid(); };
    if (!split(1))
        return 0;
    int lo = 1, hi = T;  // split(lo) holds
    if (split(hi))
        return (size_t)hi * c.top_k;
    while (hi - lo > 1) {
        const int mid = lo + (hi - lo) / 2;
        if (split(mid))
            lo = mid;
        else
            hi = mid;
    }
    return (size_t)lo * c.top_k;
}

int shared_down_parts(const moe_config_t &c)
{
    // a chunk about as long as a routed expert's reduction, and no longer than 2560 columns
    int s = c.shared_inter / c.inter;
    if (s < c.shared_inter / 2560)
        s = c.shared_inter / 2560;
    if (s < 2)
        return 1;
    return split_parts(c.shared_inter, s > 8 ? 8 : s);
}

cudaError_t launch_ffn_down(const moe_config_t &c, const moe_weights_t &w, int T, PlanView plan,
                            bool with_shared, const __nv_bfloat16 *h, const __nv_bfloat16 *h_shared,
                            __nv_bfloat16 *y, __nv_bfloat16 *y_shared, int shared_parts,
                            int routed_parts, bool f32_out, int32_t *status, cudaStream_t s)
{
    const uint64_t A = (uint64_t)T * c.top_k, H = c.hidden, E = c.n_experts;
    FfnArgs a{};
    a.rows[0] = a.rows[1] = c.hidden;
    a.K[0] = c.inter;
    a.K[1] = c.shared_inter;
    a.max_tile = routed_tile_rows(c, T, routed_parts).down;
    a.shared_ksplit = with_shared ? shared_parts : 1;
    a.shared_kchunk = with_shared ? split_chunk(c.shared_inter, a.shared_ksplit) : 128;
    a.shared_part_stride = (long long)T * c.hidden;
    a.shared_tiles = with_shared ? shared_tile_count(c, T, c.hidden, c.hidden, c.inter, c.shared_inter,
                                                     a.shared_ksplit, 128, 256)
                                 : 0;
    ffn_geometry(c, T, a);
    a.wait_us = (int)(FF_WAIT_NS / 1000ull);
    FfnMaps maps;
    const MapKey key = map_key(false, w.w_down, h, with_shared ? w.ws_down : nullptr,
                               with_shared ? h_shared : nullptr, nullptr, nullptr, nullptr, E,
                               (uint64_t)c.inter, H, A, with_shared ? (uint64_t)c.shared_inter : 0,
                               (uint64_t)T);
    if (!map_cache_lookup(key, maps)) {
        memset(&maps, 0, sizeof maps);
        bool ok = make_weight_maps(maps.w[0][0], w.w_down, E * H, c.inter) &&
                  make_weight_maps(maps.x[0], h, A, c.inter);
        if (with_shared)
            ok = ok && make_weight_maps(maps.w[1][0], w.ws_down, H, c.shared_inter) &&
                 make_weight_maps(maps.x[1], h_shared, T, c.shared_inter);
        if (!ok)
            return cudaErrorInvalidValue;
        map_cache_store(key, maps);
    }
    a.out[0] = y;
    a.out[1] = y_shared;
    a.out_ld[0] = a.out_ld[1] = c.hidden;
    a.plan_header = plan.header;
    a.seg = plan.seg;
    a.max_seg = max_segments(c.n_experts, T * c.top_k);
    a.f32_out = f32_out ? 1 : 0;
    a.claim_counter = plan.header + 3;
    a.done[0] = plan.done_routed;
    a.done[1] = plan.done_shared;
    a.routed_ksplit = routed_parts;
    a.routed_kchunk = split_chunk(c.inter, routed_parts);
    if ((long long)(routed_parts - 1) * a.routed_kchunk >= c.inter ||
        (with_shared && (long long)(a.shared_ksplit - 1) * a.shared_kchunk >= c.shared_inter))
        return cudaErrorInvalidValue;  // an empty chunk would leave its plane unwritten
    a.routed_part_stride = (long long)A * c.hidden;
    a.status = status;
    a.T = T;
    a.with_shared = with_shared ? 1 : 0;
    return ffn_pairs(c, T) ? launch_ffn<false, true>(a, maps, s) : launch_ffn<false, false>(a, maps, s);
}

}  // namespace moe
