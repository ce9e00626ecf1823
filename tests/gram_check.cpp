// Host check of the plan of the integer Gram matrix (no GPU needed): the slices of every chunk, the columns of a slice, the memory of the digits.
#include <cstdio>
#include <cstdlib>

#include "rocket_gram.h"

using namespace rocket;

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

int main() {
    const int rows[] = {1, 64, 65, 100, 128, 129, 300, 677, 897, 900, 1500, 1600, 1728, 2500, 4096};
    for (int N : rows)
        for (long long P = 1; P < 40000000ll; P += 1 + P / 7) {
            for (int p : {(int)P, N == 1728 ? 1354944 : (int)P / 64 * 64 + 1}) {
                const size_t most = P % 3 == 0 ? kGramDigitBytes / 5 : kGramDigitBytes;
                const GramPlan g = gram_plan(N, p, 148, most);
                const int blocks = (p + kGramStageK - 1) / kGramStageK;
                REQUIRE(g.chunk >= 1 && g.slices >= 1 && g.slices <= g.chunk, "%d x %d: %d slices of %d blocks", N, p, g.slices, g.chunk);
                REQUIRE(g.groups * 8 >= N && g.groups % (kGramTileM / 8) == 0, "%d x %d: %d groups", N, p, g.groups);
                const size_t block = (size_t)g.groups * kGramGroupBytes;
                REQUIRE(g.digit_bytes == g.chunk * block && (g.chunk == 1 || g.digit_bytes <= most), "%d x %d: digits", N, p);
                for (int b0 = 0; b0 < blocks; b0 += g.chunk) {
                    const int nb = blocks - b0 < g.chunk ? blocks - b0 : g.chunk, slices = gram_slices(g, nb);
                    REQUIRE(slices >= 1 && slices <= g.slices, "%d x %d: %d slices where there is room for %d", N, p, slices, g.slices);
                    for (int s = 0; s < slices; ++s) {       // the blocks that the kernel takes for slice s
                        const int n = (int)((long long)nb * (s + 1) / slices) - (int)((long long)nb * s / slices);
                        REQUIRE(n >= 1 && n <= kGramSliceStages, "%d x %d: %d blocks in slice %d of %d of a chunk of %d", N, p, n, s, slices, nb);
                    }
                }
            }
            if (failures > 20) return 1;
        }
    if (failures == 0) std::printf("ok\n");
    return failures ? 1 : 0;
}
