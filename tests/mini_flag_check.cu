// A call of the MINIROCKET transform whose wait gave up returns NaN, and no later call does.  The wait is not made to run out: the
// flag that the kernel would set is set from here, between calls.  Prints the features' bits, which must not depend on how many
// launches the batch takes.
#include <cmath>
#include <cstdio>

#include "rocket_mini.cu"

namespace rocket {
std::atomic<int64_t> g_launch_count{0}, g_alloc_count{0};
void release_cached_workspaces() {}
}

int main() {
    const int C = 3, L = 700, N = 50;
    rocket_mini_t* p = nullptr;
    std::vector<float> x((size_t)N * C * L);
    for (size_t i = 0; i < x.size(); ++i) x[i] = std::sin(0.37f * (float)i) + 0.001f * (float)(i % 97);
    if (rocket_mini_create(5, C, L, 840, &p) != ROCKET_OK || rocket_mini_fit(p, x.data(), N) != ROCKET_OK) return 2;
    float *dx = nullptr, *df = nullptr;
    const size_t values = (size_t)N * p->F;
    if (cudaMalloc(&dx, x.size() * 4) != cudaSuccess || cudaMalloc(&df, values * 4) != cudaSuccess) return 2;
    cudaMemcpy(dx, x.data(), x.size() * 4, cudaMemcpyHostToDevice);
    std::vector<float> first(values), now(values);
    auto call = [&](std::vector<float>& to) {
        const int st = rocket_mini_transform(p, dx, N, C, L, df, nullptr);
        cudaMemcpy(to.data(), df, values * 4, cudaMemcpyDeviceToHost);
        return st == ROCKET_OK && cudaGetLastError() == cudaSuccess;
    };
    if (!call(first)) return 2;
    for (float v : first) if (!(v >= 0.0f && v <= 1.0f)) { std::fprintf(stderr, "feature %g\n", v); return 1; }
    const int one = 1;
    cudaMemcpy(&p->flags[1].failed, &one, 4, cudaMemcpyHostToDevice);      // the second call's flag
    if (!call(now)) return 2;
    for (float v : now) if (!std::isnan(v)) { std::fprintf(stderr, "a call whose wait gave up returned %g\n", v); return 1; }
    for (int i = 0; i < 2 * kMFlags + 3; ++i) {
        if (!call(now)) return 2;
        for (size_t k = 0; k < values; ++k)
            if (now[k] != first[k]) { std::fprintf(stderr, "call %d after it: feature %zu is %g, was %g\n", i, k, now[k], first[k]); return 1; }
    }
    rocket_mini_destroy(p);
    unsigned long long h = 1469598103934665603ull;
    for (float v : first) { unsigned b; std::memcpy(&b, &v, 4); h = (h ^ b) * 1099511628211ull; }
    std::printf("ok %016llx\n", h);
    return 0;
}
