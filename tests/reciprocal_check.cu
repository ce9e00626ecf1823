// Quotients by way of pivot_reciprocal against correctly rounded ones, over all exponents of pivots the factorisation accepts and whose
// reciprocals are normal.  Two roundings of 2^-53 each on top of the method's 2^-60: within 2^-52 (1 + 2^-7) of x / d.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "rocket_pivot.cuh"

__global__ void quotients(const double* x, const double* d, double* q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double y, p;
    rocket::pivot_reciprocal(d[i], y, p);
    q[i] = rocket::times_reciprocal(x[i], y, p);
}

int main() {
    std::vector<double> x, d;
    uint64_t s = 88172645463325252ull;
    auto bits = [&] { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
    auto value = [](int exponent, uint64_t mantissa) {
        const uint64_t b = (uint64_t)(exponent + 1023) << 52 | (mantissa & 0xfffffffffffffull);
        double v;
        std::memcpy(&v, &b, 8);
        return v;
    };
    for (int e = -1022; e <= 1020; ++e)
        for (int i = 0; i < 260; ++i) {
            const uint64_t m = i == 0 ? 0 : i == 1 ? ~0ull : i == 2 ? 1 : i == 3 ? 0xfffff00000000ull : i == 4 ? 0x00000ffffffffull : bits();
            d.push_back(value(e, m));
            // a numerator of the pivot's size, and one: the quotient and the reciprocal itself
            x.push_back(i % 2 ? value(e, bits()) : 1.0);
        }
    const int n = (int)d.size();
    double *dx, *dd, *dq;
    std::vector<double> q(n);
    if (cudaMalloc(&dx, n * 8) != cudaSuccess || cudaMalloc(&dd, n * 8) != cudaSuccess || cudaMalloc(&dq, n * 8) != cudaSuccess) return 2;
    cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dd, d.data(), n * 8, cudaMemcpyHostToDevice);
    quotients<<<(n + 255) / 256, 256>>>(dx, dd, dq, n);
    if (cudaMemcpy(q.data(), dq, n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    double worst = 0.0;
    for (int i = 0; i < n; ++i) {
        const double want = x[i] / d[i], err = std::fabs(q[i] - want) / want;
        if (!(err <= worst)) worst = err;
        if (!(err <= std::ldexp(1.0 + 1.0 / 128.0, -52))) {
            std::fprintf(stderr, "%a / %a: %a, not %a\n", x[i], d[i], q[i], want);
            return 1;
        }
    }
    std::printf("ok: %d quotients, the worst %.3g off\n", n, worst);
    return 0;
}
