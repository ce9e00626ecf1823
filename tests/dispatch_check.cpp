// Host-side checks of the rules by which a call is handed out to the kernels (no GPU needed).
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

using namespace rocket;
using namespace rocket::fast;

namespace rocket { std::atomic<int64_t> g_launch_count{0}; }

static int failures = 0;
#define REQUIRE(cond, ...)                                            \
    do {                                                              \
        if (!(cond)) {                                                \
            std::fprintf(stderr, "FAIL line %d: ", __LINE__);          \
            std::fprintf(stderr, __VA_ARGS__);                        \
            std::fprintf(stderr, "\n");                               \
            ++failures;                                               \
        }                                                             \
    } while (0)

constexpr int kSms = 148;
constexpr int64_t kL2 = 126ll << 20;

// Every (unit, example) is in one item; the copies of an item fit the L2; warps get work enough; the soft modes' sets are long.
static void check_stream_items() {
    for (int mode = 0; mode < 4; ++mode)
        for (int N : {1, 2, 7, 24, 60, 1000})
            for (int C : {1, 12, 20, 255})
                for (int L : {1000, 50000, 100000, 200000, 1000000})
                    for (int units : {3, 400, 5000, 90000, 400000}) {
                        const StreamItems s = stream_items(N, C, L, units, 13.0 * units, mode, kSms, kL2);
                        const int64_t bytes = (int64_t)C * kWCopies * L * 4;
                        REQUIRE(s.examples >= 1 && s.examples <= N && (int64_t)s.groups * s.examples >= N && (int64_t)(s.groups - 1) * s.examples < N,
                                "items of %d examples, %d groups for %d", s.examples, s.groups, N);
                        REQUIRE(s.groups_per_set >= 1 && s.groups_per_set <= s.groups, "groups of a set");
                        REQUIRE(s.examples == 1 || s.examples * bytes <= kL2 / 2, "the copies of an item: %d x %lld", s.examples, (long long)bytes);
                        REQUIRE(s.examples == 1 || (int64_t)s.groups * units >= 12ll * kSms * kWWarps, "items per warp");
                        if (mode == 1 || mode == 2)
                            REQUIRE(s.groups_per_set == s.groups || (int64_t)s.groups_per_set * units >= (int64_t)kWSoftSetItems * kSms * kWWarps, "short set");
                        else
                            REQUIRE(s.groups_per_set == 1 || s.groups_per_set * s.examples * bytes <= kL2 / 3, "the copies of a set");
                    }
}

// The rows of a column that lie in a series, for the longest series there are: positions beyond 2^31 must not wrap.
static void check_rows_in_series() {
    const int kRows = 22;
    for (long long L : {9ll, 64ll, 50001ll, 700000000ll, 900000000ll, 1300000001ll, 2147483647ll})
        for (long long d : {1ll, 2ll, 7ll, (L - 1) / 8, (L - 1) / 9, (L - 1) / 13}) {
            if (d < 1) continue;
            const long long rows = (L + d - 1) / d;
            for (long long t0 : {-4ll, -3ll, 0ll, 10ll, rows - 30, rows - 22, rows - 21, rows - 9, rows - 1, rows + 5})
                for (long long r : {0ll, 1ll, d / 2, d - 1}) {
                    if (r >= d || t0 < -kRows || t0 > 0x7fffffffll) continue;
                    int lo, hi;
                    rows_in_series((int)t0, (int)r, (int)(L / d), (int)(L % d), kRows, lo, hi);
                    for (int s = 0; s < kRows; ++s) {
                        const long long u = (t0 + s) * d + r;
                        REQUIRE((s >= lo && s < hi) == (u >= 0 && u < L), "L %lld d %lld row %lld + %d column %lld", L, d, t0, s, r);
                    }
                }
        }
}

// A tile of the stream kernel is interior exactly when the masks of its columns say so, at every length.
static void check_tile_interior() {
    for (long long nout : {1000ll, 100000ll, 400000000ll, 700000001ll, 1073741824ll})
        for (long long d : {64ll, 65ll, 1000ll, nout / 7, nout / 6 + 1})
            for (long long p : {0ll, 4 * d, 5 * d - 3})
                for (int R : {8, 12, 16}) {
                    if (d < 64 || 7 * d > 2 * nout + 4096) continue;
                    const long long lo = -p, hi = nout - p, tl = lo >= 0 ? lo / d : -((-lo + d - 1) / d), th = hi / d;
                    if (hi < 0) continue;
                    for (long long t : {tl, tl + 1, 0ll, th - R - 1, th - R, th - R + 1, th - 1})
                        for (long long c0 : {0ll, 64ll, (d - 1) / 64 * 64}) {
                            bool all = true;
                            for (int l = 0; l < 64; ++l) {
                                int a, b;
                                valid_rows_tc((int)t, (int)(c0 + l), (int)tl, (int)(lo - tl * d), (int)th, (int)(hi - th * d), R, c0 + l < d, a, b);
                                all = all && a == 0 && b == R;
                            }
                            REQUIRE(tile_interior((int)t, (int)c0, w_span(R, (int)d), (int)d, (int)lo, (int)hi) == all, "nout %lld d %lld p %lld R %d row %lld column %lld",
                                    nout, d, p, R, t, c0);
                        }
                }
}

// The copies of a pass stay within their budget, whatever the channels and the length, and shrink to what there is room for.
static void check_copies() {
    for (int C : {1, 3, 20, 32, 255})
        for (int64_t pitch : {1000ll, 110000ll, 440000ll, 2200000ll, 220000000ll}) {
            const int n = stream_chunk(C, pitch);
            const int64_t example = 4 * kWCopies * (int64_t)C * pitch;
            REQUIRE(n >= 1 && (n == 1 || n * example <= std::max<int64_t>(kWCopyBytes, kWMostCopyBytes)), "%d examples of %lld", n, (long long)example);
            REQUIRE(n <= kWFewExamples || n * example <= kWCopyBytes, "%d examples of %lld", n, (long long)example);
        }
    REQUIRE(stream_chunk(20, 108416) == 13 && stream_chunk(20, 433440) == 4, "the benchmark's lengths");
    for (int room : {0, 1, 2, 5, 12, 13, 40}) {
        int tries = 0;
        const int got = fit_examples(13, [&](int n) { ++tries; return n <= room; });
        REQUIRE(got <= room && (got > 0) == (room > 0) && (room < 13 || got == 13) && tries <= 4 && (room < 1 || got > room / 4), "%d of %d", got, room);
    }
}

static PlanHost plan_of(int C, int L, int K, bool only_used = true) {
    HostParams hp;
    generate_host_params(8527, K, C, L, hp);
    hp.channel_offset.assign(hp.K + 1, 0);
    hp.weight_offset.assign(hp.K + 1, 0);
    for (int k = 0; k < hp.K; ++k) {
        hp.channel_offset[k + 1] = hp.channel_offset[k] + hp.num_channels[k];
        hp.weight_offset[k + 1] = hp.weight_offset[k] + hp.num_channels[k] * hp.length[k];
    }
    PlanHost plan;
    build_plan(hp, kSplitDefault, plan, false, only_used);
    return plan;
}

// Many channels: the generic kernels where they were measured to be faster, the fused ones where those were; handles whose examples the resident
// kernel holds are not asked.
static void check_generic() {
    struct Case { int N, C, L, K, generic, asked; };
    for (const Case& c : {Case{1, 32, 32, 1500, 1, 0}, Case{1, 21, 100, 300, 1, 0}, Case{32, 255, 102, 1500, 1, 0}, Case{32, 255, 1002, 60, 1, 1}, Case{1, 64, 31, 300, 1, 0},
                          Case{6, 32, 102, 1500, 1, 0}, Case{24, 32, 1751, 2000, 0, 0}, Case{1, 32, 4000, 300, 0, 1}, Case{32, 255, 4002, 1500, 0, 1}, Case{6, 64, 4000, 60, 0, 1},
                          Case{32, 21, 300, 1500, 0, 0}, Case{1, 30, 100000, 100, 0, 1}, Case{4, 100, 20000, 500, 0, 1}, Case{32, 64, 4003, 60, 0, 1}, Case{32, 32, 4000, 60, 0, 1}}) {
        // as a handle has it, and with every plan: the rule is asked for backwards that the resident kernel does not serve
        REQUIRE(always_fused(plan_of(c.C, c.L, c.K), c.C, false) == (c.asked == 0), "%d x %d x %d, %d kernels", c.N, c.C, c.L, c.K);
        const PlanHost plan = plan_of(c.C, c.L, c.K, false);
        REQUIRE(generic_pays(plan, c.N, kSms, false) == (c.generic != 0), "%d x %d x %d, %d kernels", c.N, c.C, c.L, c.K);
        for (int way = 0; way < 4; ++way)
            for (int most : {1, 7, 32, 300}) {
                const bool generic = (way & 1) != 0, soft = (way & 2) != 0;
                const int up_to = pays_up_to(plan, most, kSms, soft, generic);
                for (int n = 1; n <= most; ++n)
                    REQUIRE(n <= up_to || generic_pays(plan, n, kSms, soft) != generic, "%d of at most %d examples", n, up_to);
            }
    }
}

// Hard transforms of short series that go to the tile kernels: their handles hold both plans, others what their calls use.
static void check_tiles_from() {
    struct Case { int C, L, K, from; };
    for (const Case& c : {Case{6, 1400, 20000, 60}, Case{6, 1344, 20000, 0}, Case{6, 1400, 9999, 0}, Case{2, 1400, 20000, 0}, Case{2, 2100, 10000, 60},
                          Case{3, 2049, 30000, 20}, Case{6, 2048, 30000, 40}, Case{5, 1501, 20000, 0}, Case{3, 1500, 20000, 60}, Case{1, 2100, 20000, 0}, Case{20, 1345, 20000, 60}, Case{32, 1700, 20000, 0}, Case{3, 6000, 20000, 0}}) {
        const PlanHost plan = plan_of(c.C, c.L, c.K);
        REQUIRE(plan.r_tiles_from == c.from, "%d x %d, %d kernels: from %d examples", c.C, c.L, c.K, plan.r_tiles_from);
        REQUIRE(c.from == 0 || (plan.resident && !plan.sitems.empty() && !plan.wunits.empty()), "%d x %d: both plans", c.C, c.L);
        REQUIRE(c.from == 0 || (resident_forward(plan, c.from - 1, true) && !resident_forward(plan, c.from, true) && resident_forward(plan, c.from, false)), "%d x %d", c.C, c.L);
        REQUIRE(c.from != 0 || resident_forward(plan, 1 << 20, true) == plan.resident, "%d x %d", c.C, c.L);
    }
    REQUIRE(plan_of(6, 1400, 9999).sitems.empty(), "tiles that no call uses");
}

// Kernels from standard input (C, L, K, then per kernel length, dilation, padding and its channels): prints, for N examples and the plan a handle
// has, how many examples the small-dilation tiles of each class share and how many tiles there are of each, and which kernels serve the
// forward modes and the backward: g(eneric), r(esident) or t(iles).
static int print_sharing(int N) {
    HostParams hp;
    if (std::scanf("%d %d %d", &hp.C, &hp.L, &hp.K) != 3) return 2;
    hp.channel_offset.assign(1, 0);
    hp.weight_offset.assign(1, 0);
    for (int k = 0; k < hp.K; ++k) {
        int len, d, p, m, c;
        if (std::scanf("%d %d %d %d", &len, &d, &p, &m) != 4) return 2;
        hp.length.push_back(len); hp.dilation.push_back(d); hp.padding.push_back(p); hp.num_channels.push_back(m);
        for (int q = 0; q < m && std::scanf("%d", &c) == 1; ++q) hp.channel_idx.push_back(c);
        hp.channel_offset.push_back((int)hp.channel_idx.size());
        hp.weight_offset.push_back(hp.weight_offset.back() + m * len);
        hp.bias.push_back(0.5f);
    }
    hp.weights.assign(hp.weight_offset.back(), 1.0f);
    PlanHost plan;
    build_plan(hp, kSplitDefault, plan, false, true);
    const SGroups s = s_groups(plan, N, kSms);
    for (int i = 0; i < 3; ++i) std::printf("%d %d ", s.examples[i], s.end[i] - (i ? s.end[i - 1] : 0));
    auto served = [&](bool hard, bool soft, bool backward) {
        if (!always_fused(plan, hp.C, backward) && generic_pays(plan, N, kSms, soft)) return 'g';
        return (backward ? resident_backward(plan) : resident_forward(plan, N, hard)) ? 'r' : 't';
    };
    std::printf("%c%c%c\n", served(true, false, false), served(false, true, false), served(false, true, true));
    return 0;
}

int main(int argc, char** argv) {
    if (argc > 1) return print_sharing(std::atoi(argv[1]));
    check_copies();
    check_tile_interior();
    check_rows_in_series();
    check_stream_items();
    check_generic();
    check_tiles_from();
    if (failures == 0) std::printf("ok\n");
    return failures ? 1 : 0;
}
