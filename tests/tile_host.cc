// The host's choice of workers and of the routed tiles' height (csrc/ffn_geometry.h) on a device of
// 148 SMs, for calls read from the standard input, one a line:
//   experts top_k hidden inter shared_inter tokens MOE_FF_WIDE MOE_FF_PAIR   (WIDE -1: unset)
// prints, a line each: CTAs per worker, weight rows per CTA and tile of the gate/up and of the
// (unsplit) down pass, CTAs per SM of a large layer call's row gather.
#include <stdint.h>
#include <stdio.h>

#include <algorithm>

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

static int g_wide, g_pair;
int moe::sm_count() { return 148; }
int moe::geometry_override() { return g_wide; }
bool moe::pairs_forced() { return g_pair; }

int main()
{
    moe_config_t c{};
    int T;
    while (scanf("%d %d %d %d %d %d %d %d", &c.n_experts, &c.top_k, &c.hidden, &c.inter, &c.shared_inter, &T,
                 &g_wide, &g_pair) == 8) {
        const TileRows t = routed_tile_rows(c, T, 1);
        printf("%d %d %d %d\n", ffn_workers(c, T).ctas, t.up, t.down,
               gather_ctas_per_sm(c, T, c.shared_inter > 0));
    }
    return 0;
}
