// Host-side check of the small-dilation tiles whose bands have fewer rows than 24 (no GPU needed): replays, with the kernel's own index
// arithmetic, which outputs the threads of every tile own.  Every output of every kernel of a small dilation is owned once, tiles marked as
// interior need no tests, and every height there is gets chosen.  With arguments C, L and kernels from standard input (K, then per kernel length,
// dilation, padding and its channels): prints the rows of a band.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

using namespace rocket;
using namespace rocket::fast;

namespace rocket { std::atomic<int64_t> g_launch_count{0}; }

#define REQUIRE(cond, ...)                                        \
    do {                                                          \
        if (!(cond)) {                                            \
            std::fprintf(stderr, "FAIL %s:%d: ", __FILE__, __LINE__); \
            std::fprintf(stderr, __VA_ARGS__);                    \
            std::fprintf(stderr, "\n");                           \
            std::exit(1);                                         \
        }                                                         \
    } while (0)

static void offsets(HostParams& hp) {
    hp.channel_offset.assign(hp.K + 1, 0);
    hp.weight_offset.assign(hp.K + 1, 0);
    for (int k = 0; k < hp.K; ++k) {
        hp.channel_offset[k + 1] = hp.channel_offset[k] + hp.num_channels[k];
        hp.weight_offset[k + 1] = hp.weight_offset[k] + hp.num_channels[k] * hp.length[k];
    }
}

static int check(int K, int C, int L) {
    HostParams hp;
    generate_host_params(11 + L, K, C, L, hp);
    offsets(hp);
    PlanHost plan;
    build_plan(hp, kSplitDefault, plan, false);
    const int R = plan.s_rows;
    std::map<int, std::vector<int>> owned;
    for (const SItem& it : plan.sitems) {
        const SBucket& b = plan.sb[it.bucket];
        for (int f = b.kbeg; f < b.kend; ++f) {
            const KRec& k = plan.krec[f];
            std::vector<int>& mine = owned[f];
            mine.resize(k.nout, 0);
            REQUIRE(k.len + R - 1 <= b.rows && b.rows <= kSRowsMax, "rows of a tile");
            for (int c = it.c0; c < it.c0 + kWarpCols; ++c) {
                const int band = c / b.d, u0 = s_column_u0(b, c, R);
                int lo, hi;
                valid_rows_tc(b.tmin + band * R, c - band * b.d, k.tl, k.rl, k.th, k.rh, R, c < b.raster_len, lo, hi);
                if (it.interior) REQUIRE(lo == 0 && hi == R, "interior tile");
                for (int o = lo; o < hi; ++o) {
                    const int i = u0 + o * b.d + k.p;
                    REQUIRE(i >= 0 && i < k.nout, "output %d of %d", i, k.nout);
                    ++mine[i];
                }
            }
        }
    }
    for (auto& kv : owned)
        for (int n : kv.second) REQUIRE(n == 1, "an output of record %d owned %d times", kv.first, n);
    return R;
}

int main(int argc, char** argv) {
    if (argc > 2) {
        HostParams hp;
        hp.C = std::atoi(argv[1]); hp.L = std::atoi(argv[2]);
        if (std::scanf("%d", &hp.K) != 1) return 2;
        for (int k = 0; k < hp.K; ++k) {
            int len, d, p, m, c;
            if (std::scanf("%d %d %d %d", &len, &d, &p, &m) != 4) return 2;
            hp.length.push_back(len); hp.dilation.push_back(d); hp.padding.push_back(p); hp.num_channels.push_back(m);
            for (int q = 0; q < m && std::scanf("%d", &c) == 1; ++q) hp.channel_idx.push_back(c);
            hp.bias.push_back(0.5f);
        }
        offsets(hp);
        hp.weights.assign(hp.weight_offset.back(), 1.0f);
        PlanHost plan;
        build_plan(hp, kSplitDefault, plan, false);
        std::printf("%d %d\n", plan.s_rows, plan.resident ? 1 : 0);
        return 0;
    }
    std::map<int, int> chosen;
    for (int L : {1000, 2301, 3000, 3100, 3207, 3700, 5000, 5501, 7001, 13000})
        for (int C : {1, 6, 20}) ++chosen[check(150, C, L)];
    for (int R : {kRS, kSLowRows[0], kSLowRows[1]}) REQUIRE(chosen[R] > 0, "%d rows are never chosen", R);
    std::printf("ok\n");
    return 0;
}
