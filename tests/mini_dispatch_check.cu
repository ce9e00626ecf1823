// Prints, for (channels, steps, features, examples) from standard input, whether the kernel that takes one combination at a time serves
// the call (148 SMs; no GPU needed).
#include <cstdio>

#include "rocket_mini.cu"

namespace rocket {
std::atomic<int64_t> g_launch_count{0}, g_alloc_count{0};
void release_cached_workspaces() {}
}

int main() {
    int C, L, F, N;
    while (std::scanf("%d %d %d %d", &C, &L, &F, &N) == 4) {
        rocket_mini_t* p = nullptr;
        if (rocket_mini_create(8527, C, L, F, &p) != ROCKET_OK) return 1;
        std::printf("%d\n", mini_walks(*p, N, 148) ? 1 : 0);
        rocket_mini_destroy(p);
    }
    return 0;
}
