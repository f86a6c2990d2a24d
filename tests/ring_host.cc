// The FFN kernels' token ring and k-step barriers, the kernels' own placement and release rule
// (TokenRing, XRingWalk in csrc/ffn_walk.cuh) in the geometries the host's own rule gives
// (csrc/ffn_geometry.h), replayed in random order on the CPU: the producers and the issuer never
// stall, agree on every position, and no live entry, weight slot or barrier pair is reused.
//
//   ring_host SEED TRIALS
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <random>
#include <vector>

#define __device__
#define __forceinline__ inline
using std::max;
using std::min;

// what the walk in the same header needs; nothing here calls it
struct __nv_bfloat16;
struct alignas(16) int4 {
    int x, y, z, w;
};
struct Dim {
    int x;
};
static Dim threadIdx, blockIdx, gridDim;
bool __all_sync(uint32_t, bool);
void __syncwarp();
void __threadfence_block();
void griddep_wait();
int atomicAdd(int32_t *, int);
int peek(const int32_t *);
void mbar_arrive(uint32_t);
void mbar_arrive_cluster(uint32_t);
void st_cluster_v4(uint32_t, int, int, int, int);
template <bool CLUSTER = false>
bool mbar_wait(uint32_t, uint32_t, volatile int *, int32_t *);

#include "ffn_geometry.h"

using namespace moe;

static int g_wide = -1, g_pair = 0;
int moe::sm_count() { return 148; }
int moe::geometry_override() { return g_wide; }
bool moe::pairs_forced() { return g_pair; }

#define CHECK(cond)                                                                               \
    do {                                                                                          \
        if (!(cond)) {                                                                            \
            printf("E=%d k=%d T=%d wide=%d pair=%d step %d, line %d: %s\n", c.n_experts, c.top_k, T, \
                   g_wide, g_pair, consumed, __LINE__, #cond);                                    \
            exit(1);                                                                              \
        }                                                                                         \
    } while (0)

template <bool PAIR>
static void replay(const moe_config_t &c, int T, const FfnArgs &a, std::mt19937 &g)
{
    auto in = [&](int lo, int hi) { return lo + (int)(g() % (unsigned)(hi - lo + 1)); };
    int consumed = 0;
    // the rings fit, an entry fits, and there is a barrier pair per weight slot
    CHECK(a.x_units * FF_X_UNIT + a.n_w_slots * a.w_slot_bytes + 1024 <= FF_SMEM_LIMIT - 512);
    CHECK(a.n_w_slots >= 2 && a.n_w_slots <= FF_STEPS);
    std::vector<int> sizes;  // one entry per k step, the same for all steps of an item
    while (sizes.size() < 60) {
        int n;
        if (c.shared_inter > 0 && in(0, 2) == 0) {
            const int nseg = (T + a.shared_seg - 1) / a.shared_seg, rows = balanced_segment_rows(T, nseg);
            CHECK(rows <= a.shared_seg);
            n = min(rows, T - in(0, nseg - 1) * rows);
        } else {  // a group of any size up to all tokens
            const int all = in(1, T), nseg = (all + a.seg_rows - 1) / a.seg_rows;
            const int rows = balanced_segment_rows(all, nseg);
            CHECK(rows <= a.seg_rows);
            n = min(rows, all - in(0, nseg - 1) * rows);
        }
        CHECK(n > 0);
        const int m = token_pieces<PAIR>(n) * a.kboxes;
        CHECK(m <= a.x_units);
        sizes.insert(sizes.end(), in(1, 6), m);
    }
    const int steps = (int)sizes.size();
    TokenRing producer(a.x_units);
    XRingWalk issuer(a.x_units);
    int starts[FF_STEPS], x_issued = 0, w_issued = 0;
    std::vector<int> at(steps, -1);
    while (consumed < steps) {
        bool can[3] = {x_issued < steps, w_issued < steps && w_issued < consumed + a.n_w_slots,
                       consumed < x_issued && consumed < w_issued};
        const int order = in(0, 5), first = order % 3, second = (first + 1 + order / 3) % 3;
        const int tries[3] = {first, second, 3 - first - second};
        bool moved = false;
        for (int who : tries) {
            if (!can[who] || moved)
                continue;
            if (who == 0) {  // token producer: one step of it (a placed entry waits for room)
                if (at[x_issued] < 0)
                    at[x_issued] = producer.place(sizes[x_issued]);
                if (producer.must_release()) {
                    if (consumed <= producer.released)
                        continue;  // the wait
                    producer.release(starts);
                } else {
                    const int j = x_issued, lo = at[j], hi = lo + sizes[j];
                    CHECK(lo >= 0 && hi <= a.x_units && j - consumed < FF_STEPS);
                    for (int q = consumed; q < j; ++q)
                        CHECK(hi <= at[q] || at[q] + sizes[q] <= lo);
                    producer.issued(starts);
                    ++x_issued;
                }
            } else if (who == 1) {  // weight producer: slot and barrier pair are free
                CHECK(w_issued - consumed < FF_STEPS);
                ++w_issued;
            } else {  // issuer: reads the entry where it says it lies
                CHECK(issuer.place(sizes[consumed]) == at[consumed]);
                ++consumed;
            }
            moved = true;
        }
        CHECK(moved);  // else every role waits for another
    }
}

int main(int argc, char **argv)
{
    if (argc != 3)
        return 2;
    std::mt19937 g((unsigned)atoi(argv[1]));
    const int shapes[][5] = {  // experts, top_k, hidden, inter, shared_inter
        {8, 2, 256, 512, 0},       {60, 4, 2048, 1408, 5632}, {64, 8, 3584, 2560, 20480},
        {8, 2, 4096, 14336, 0},    {256, 8, 7168, 2048, 2048}, {1, 1, 3584, 20480, 20480},
        {24, 16, 160, 224, 96},    {4, 2, 544, 96, 0}};
    const int tokens[] = {1, 2, 16, 17, 33, 63, 64, 65, 80, 127, 128, 129, 192, 255, 256, 257, 320, 640, 1280, 4096};
    long single = 0, pairs = 0, rings[97] = {};
    for (int trial = 0; trial < atoi(argv[2]); ++trial)
        for (const auto &s : shapes)
            for (int T : tokens) {
                moe_config_t c{};
                c.n_experts = s[0], c.top_k = s[1], c.hidden = s[2], c.inter = s[3], c.shared_inter = s[4];
                g_wide = trial % 4 < 2 ? -1 : trial % 4 - 2;
                g_pair = trial % 3 == 2;
                FfnArgs a{};
                ffn_geometry(c, T, a);
                if (!ffn_pairs(c, T) && (a.seg_rows != FF_SEG || a.kboxes != 2 || a.acc_sets != 2))
                    return printf("T=%d: not the geometry the single-CTA kernels are built for\n", T), 1;
                ++rings[a.x_units];
                if (ffn_pairs(c, T))
                    ++pairs, replay<true>(c, T, a, g);
                else
                    ++single, replay<false>(c, T, a, g);
            }
    printf("rings hold: %ld single, %ld pairs; units 16: %ld, 32: %ld, 48: %ld\n", single, pairs, rings[16],
           rings[32], rings[48]);
    return 0;
}
