// Host-side checks of the rules by which a call is handed out to the kernels (no GPU needed).
#include <cstdio>

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

int main() {
    check_stream_items();
    if (failures == 0) std::printf("ok\n");
    return failures ? 1 : 0;
}
