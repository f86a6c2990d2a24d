// The FFN kernels' work walk (csrc/ffn_walk.cuh) run on host threads: two lanes of every warp of
// a few workers (CTAs, or pairs of CTAs), with barriers, votes and cluster stores standing in for
// the hardware's.  Every walked item is checked: all lanes and roles of a worker see the same ones,
// and together the workers cover every piece of work exactly once.
//
// The stand-ins order memory no more than the originals are documented to: a warp vote makes the
// lanes agree but is a relaxed atomic; __syncwarp and the barriers release and acquire.  Built with
// -fsanitize=thread the program therefore also finds a hand-over that relies on anything less.
//
//   walk_host SEED TRIALS
#include <sched.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <map>
#include <memory>
#include <random>
#include <set>
#include <thread>
#include <tuple>
#include <vector>

#define __device__
#define __forceinline__ inline
using std::max;
using std::min;

struct __nv_bfloat16;
struct alignas(16) int4 {
    int x, y, z, w;
};
struct Dim {
    int x;
};

constexpr int LANES = 2;  // simulated lanes of a warp
constexpr int ROUNDS = 1024;

struct Rendezvous {  // a counter per round, cleared half the ring ahead
    std::atomic<uint32_t> slot[ROUNDS] = {};
    uint32_t meet(uint32_t round, uint32_t add, std::memory_order rmw, std::memory_order ld)
    {
        std::atomic<uint32_t> &s = slot[round % ROUNDS];
        s.fetch_add(add, rmw);
        uint32_t v;
        while (((v = s.load(ld)) & 255u) != (uint32_t)LANES)
            sched_yield();
        slot[(round + ROUNDS / 2) % ROUNDS].store(0, std::memory_order_relaxed);
        return v;
    }
};
struct Warp {
    Rendezvous vote, sync;
};

static thread_local Dim threadIdx, blockIdx, gridDim;
static thread_local Warp *t_warp;
static thread_local uint32_t t_votes, t_syncs;
static std::atomic<int> g_failed{0};

static bool __all_sync(uint32_t, bool pred)
{
    return (t_warp->vote.meet(t_votes++, pred ? 1u : 257u, std::memory_order_relaxed, std::memory_order_relaxed) >> 8) == 0;
}
static void __syncwarp()
{
    t_warp->sync.meet(t_syncs++, 1u, std::memory_order_acq_rel, std::memory_order_acquire);
}
static void __threadfence_block() {}
static void griddep_wait() {}
static int atomicAdd(int32_t *p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_RELAXED); }
static int peek(const int32_t *p) { return __atomic_load_n(p, __ATOMIC_RELAXED); }

struct Barrier {
    uint32_t count = 1;
    std::atomic<uint32_t> arrived{0};
};
static std::vector<std::unique_ptr<Barrier>> g_bars;  // barrier i at "shared address" 8 * i
static std::vector<int> g_arena;                      // ring entries; address = byte offset

static void mbar_arrive(uint32_t bar) { g_bars[bar / 8]->arrived.fetch_add(1, std::memory_order_acq_rel); }
static void mbar_arrive_cluster(uint32_t bar) { mbar_arrive(bar); }
static void st_cluster_v4(uint32_t addr, int a, int b, int c, int d)
{
    int *p = g_arena.data() + addr / 4;
    p[0] = a, p[1] = b, p[2] = c, p[3] = d;
}
template <bool CLUSTER = false>
static bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *, int32_t *)
{
    Barrier &b = *g_bars[bar / 8];
    const auto t0 = std::chrono::steady_clock::now();
    while ((b.arrived.load(std::memory_order_acquire) / b.count & 1u) == parity) {
        sched_yield();
        if (std::chrono::steady_clock::now() - t0 > std::chrono::seconds(20)) {
            g_failed = 1;
            return false;
        }
    }
    return true;
}

#include "ffn_walk.cuh"

using namespace moe;

// what an item covers: group kind, expert, weight rows, token rows, reduction range, plane
using Key = std::tuple<int, int, int, int, int, int, int, int, int, int, long long>;
static Key key_of(const Item &it)
{
    return Key(it.grp, it.expert, it.f0, it.h, it.row0, it.n, it.seg, it.w_once, it.k0, it.k1, it.out_off);
}

#define CHECK(cond)                                              \
    do {                                                         \
        if (!(cond)) {                                           \
            printf("trial %d, line %d: %s\n", g_trial, __LINE__, #cond); \
            exit(1);                                             \
        }                                                        \
    } while (0)
static int g_trial;

struct Rng {
    std::mt19937 g;
    int pick(std::initializer_list<int> v) { return v.begin()[g() % v.size()]; }
    int in(int lo, int hi) { return lo + (int)(g() % (unsigned)(hi - lo + 1)); }
};

template <bool PAIR>
static void trial(Rng &rng)
{
    constexpr int CTAS = PAIR ? 2 : 1, UNIT = 16 * CTAS;
    const bool down = rng.in(0, 1);
    FfnArgs a{};
    a.seg_rows = PAIR && rng.in(0, 1) ? 256 : 128;
    const int full = down ? 256 : 128;  // rows of a full tile; the routed ones may be lower
    a.max_tile = rng.pick({full / 2, full});
    a.rows[0] = rng.pick({32, 96, 224, 288, 544, 1088});
    a.rows[1] = down ? a.rows[0] : rng.pick({32, 96, 704, 1408});
    a.K[0] = rng.pick({32, 96, 512, 1056});
    a.K[1] = down ? rng.pick({32, 160, 1408}) : a.K[0];
    a.T = rng.pick({1, 5, 64, 65, 128, 129, 300, 513});
    a.with_shared = rng.in(0, 2) > 0;
    a.first_fixed = !down;
    auto split = [&](int K, int parts, int &chunk) {  // as the host cuts a reduction
        chunk = ((K + parts - 1) / parts + 127) / 128 * 128;
        return (K + chunk - 1) / chunk;
    };
    a.routed_ksplit = split(a.K[0], down ? rng.in(1, 4) : 1, a.routed_kchunk);
    a.shared_ksplit = split(a.K[1], down ? rng.in(1, 3) : 1, a.shared_kchunk);
    a.routed_part_stride = 1000000;
    a.shared_part_stride = 10000000;
    a.shared_seg = a.T > 64 && a.T <= 128 && rng.in(0, 1) ? 64 : a.seg_rows;
    const int most[2] = {a.max_tile >> 4, full >> 4};  // units per routed and per shared tile at most
    const int s_units = a.rows[1] / UNIT;
    a.shared_tiles = a.with_shared ? rng.in((s_units + most[1] - 1) / most[1], s_units) : 0;

    std::vector<int> groups;
    for (int i = rng.in(1, 7); i > 0; --i)
        groups.push_back(rng.pick({1, 5, 16, 100, 128, 129, 200, 256, 257, 400}));
    std::vector<Segment> seg;
    int row = 0;
    for (size_t e = 0; e < groups.size(); ++e) {
        const int n = groups[e], ns = (n + a.seg_rows - 1) / a.seg_rows, first = (int)seg.size();
        for (int q = 0; q < ns; ++q) {
            seg.push_back(Segment{(int)(3 * e + 1), row, n, first, first + q, {0, 0, 0}});
        }
        row += n;
    }
    alignas(16) int32_t header[16] = {(int)seg.size(), 0, 0, 0};
    a.plan_header = header;
    a.seg = seg.data();
    a.max_seg = (int)seg.size();
    a.claim_counter = header + (down ? 3 : 2);

    // roles: the weight producer's warp and R readers in every CTA
    const int R = 2, workers = rng.in(1, 3), ctas = workers * CTAS;
    g_bars.clear();
    g_arena.assign((size_t)ctas * FF_CLAIMS * FF_CLAIM_WORDS, 0x7f7f7f7f);
    for (int c = 0; c < ctas; ++c)
        for (int i = 0; i < 2 * FF_CLAIMS; ++i) {  // full, empty (a pair's: the leader's)
            g_bars.emplace_back(new Barrier);
            if (i >= FF_CLAIMS)
                g_bars.back()->count = PAIR ? 2 * R + 1 : R;
        }
    struct Role {
        int cta, warp;
        Warp w;
        std::vector<Item> items[LANES];
    };
    std::vector<std::unique_ptr<Role>> roles;
    for (int c = 0; c < ctas; ++c)
        for (int w = 0; w <= R; ++w) {
            roles.emplace_back(new Role);
            roles.back()->cta = c;
            roles.back()->warp = w;
        }
    auto run = [&](Role *r, int lane) {
        threadIdx.x = 32 * r->warp + lane;
        blockIdx.x = r->cta;
        gridDim.x = ctas;
        t_warp = &r->w;
        t_votes = t_syncs = 0;
        const int rank = r->cta % CTAS, leader = r->cta - rank, peer = PAIR ? r->cta ^ 1 : r->cta;
        const uint32_t ring_bytes = FF_CLAIMS * FF_CLAIM_WORDS * 4, bar_bytes = 2 * FF_CLAIMS * 8;
        int abort_flag[2] = {0, 0};
        ClaimRing ring{g_arena.data() + r->cta * ring_bytes / 4, r->cta * bar_bytes,
                       r->cta * bar_bytes + 8 * FF_CLAIMS, abort_flag, nullptr, peer * ring_bytes,
                       peer * bar_bytes, leader * bar_bytes + 8 * FF_CLAIMS};
        ItemWalk<PAIR> walk(a, ring, r->warp == 0 && rank == 0, down);
        Item it;
        while (walk.next(it))
            r->items[lane].push_back(it);
    };
    std::vector<std::thread> threads;
    for (auto &r : roles)
        for (int lane = 0; lane < LANES; ++lane)
            threads.emplace_back(run, r.get(), lane);
    for (std::thread &t : threads)
        t.join();
    CHECK(!g_failed);

    // all lanes and roles of a worker walked the same items
    std::vector<Item> all;
    for (int w = 0; w < workers; ++w) {
        const std::vector<Item> &want = roles[(size_t)w * CTAS * (R + 1)]->items[0];
        for (int i = 0; i < CTAS * (R + 1); ++i)
            for (int lane = 0; lane < LANES; ++lane) {
                const std::vector<Item> &got = roles[(size_t)w * CTAS * (R + 1) + i]->items[lane];
                CHECK(got.size() == want.size());
                for (size_t q = 0; q < got.size(); ++q)
                    CHECK(key_of(got[q]) == key_of(want[q]));
            }
        all.insert(all.end(), want.begin(), want.end());
    }
    // every (kind, expert, unit of weight rows, segment, k chunk) exactly once
    std::set<std::tuple<int, int, int, int, int>> seen;
    for (const Item &it : all) {
        const int g = it.grp, chunk = g ? a.shared_kchunk : a.routed_kchunk;
        CHECK(it.h > 0 && it.h % UNIT == 0 && it.f0 % UNIT == 0 && it.h <= most[g] * UNIT);
        CHECK(it.f0 + it.h <= a.rows[g]);
        CHECK(it.k0 % 128 == 0 && it.k0 < it.k1 && it.k1 == min(a.K[g], it.k0 + chunk));
        const int part = it.k0 / chunk;
        CHECK(it.k0 % chunk == 0 && it.out_off == part * (g ? a.shared_part_stride : a.routed_part_stride));
        CHECK(it.n > 0 && it.n <= (g ? a.shared_seg : a.seg_rows));
        for (int u = it.f0; u < it.f0 + it.h; u += UNIT)
            CHECK(seen.insert({g, it.expert, u, it.seg, part}).second);
    }
    const size_t shared_segs = a.with_shared ? (a.T + a.shared_seg - 1) / a.shared_seg : 0;
    CHECK(seen.size() == seg.size() * (a.rows[0] / UNIT) * a.routed_ksplit +
                             shared_segs * s_units * a.shared_ksplit);
    // a segment's token rows are the same in all its items, its group's rows in plan order
    std::map<std::pair<int, int>, std::pair<int, int>> rows;
    for (const Item &it : all) {
        const auto at = rows.insert({{it.grp, it.seg}, {it.row0, it.n}}).first;
        CHECK(at->second == std::make_pair(it.row0, it.n));
    }
    int next[2] = {0, 0};
    for (const auto &r : rows) {
        CHECK(r.second.first == next[r.first.first]);
        next[r.first.first] += r.second.second;
    }
    CHECK(next[0] == row && (!a.with_shared || next[1] == a.T));
}

int main(int argc, char **argv)
{
    if (argc != 3)
        return 2;
    Rng rng{std::mt19937((unsigned)atoi(argv[1]))};
    for (g_trial = 0; g_trial < atoi(argv[2]); ++g_trial) {
        if (g_trial % 2)
            trial<true>(rng);
        else
            trial<false>(rng);
    }
    printf("walks agree\n");
    return 0;
}
