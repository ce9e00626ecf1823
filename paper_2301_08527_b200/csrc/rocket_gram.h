// Gram matrix of the centred features in integers on the tensor cores (rocket_gram.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace rocket {

constexpr int kGramDigits = 7, kGramTileM = 128, kGramTileN = 64, kGramStageK = 64;   // of a row; rows and columns of a tile; columns of a stage
constexpr int kGramGroupBytes = kGramDigits * 8 * kGramStageK;      // digits of eight rows and a stage
constexpr size_t kGramDigitBytes = (size_t)112 << 20;   // digits of as many columns at a time, unless that is too much memory
constexpr int kGramSliceStages = 16384 / kGramStageK;   // of a slice: a 32-bit sum holds as many columns

struct GramPlan {
    int groups, blocks_mn;     // groups of 8 rows; 128 x 64 tiles of the lower triangle
    int chunk, slices;         // blocks of 64 columns whose digits are held at a time; slices of partial tiles
    size_t digit_bytes;
};

inline GramPlan gram_plan(int N, int P, int sms, size_t most_digit_bytes = kGramDigitBytes) {
    GramPlan g{};
    g.groups = (N + kGramTileM - 1) / kGramTileM * (kGramTileM / 8);
    const int nt = (N + 63) / 64, last = (N + kGramTileM - 1) / kGramTileM - 1;
    g.blocks_mn = last * (last + 1) + std::min(2 * last + 2, nt);
    const size_t block_bytes = (size_t)g.groups * kGramGroupBytes;
    const int blocks = (P + kGramStageK - 1) / kGramStageK;
    g.chunk = (int)std::max<size_t>(1, std::min<size_t>(blocks, most_digit_bytes / block_bytes));
    g.chunk = (blocks + (blocks + g.chunk - 1) / g.chunk - 1) / ((blocks + g.chunk - 1) / g.chunk);   // evenly
    // Slices of a chunk: the fewest clocks, where a stage takes 4,800 and a block's beginning and end 10,000; no more columns than 32-bit sums
    // hold each, and 24 MB of partial tiles (or one slice).
    const size_t slice_bytes = (size_t)nt * (nt + 1) / 2 * 4096 * sizeof(double);
    const int least = (g.chunk + kGramSliceStages - 1) / kGramSliceStages, most = std::max<int>(least, std::min<int>(16, (int)(((size_t)24 << 20) / slice_bytes)));
    double best = 1e300;
    for (int s = least; s <= most && s <= g.chunk; ++s) {
        const double t = (double)(((long long)g.blocks_mn * s + sms - 1) / sms) * ((g.chunk + s - 1) / s * 4800.0 + 10000.0);
        if (t < best) { best = t; g.slices = s; }
    }
    g.digit_bytes = (size_t)g.chunk * block_bytes;
    return g;
}

// Slices of a chunk of `blocks` blocks: the last chunk may have fewer blocks than the others have slices, and a slice without a block would
// add what its accumulators held before.
inline int gram_slices(const GramPlan& g, int blocks) { return std::min(g.slices, blocks); }

// Partial tiles part[slices][tiles of the lower triangle, 64 x 64][64][64] of Fc Fc^T.  up, down: N doubles each; digits: digit_bytes, 128-byte
// aligned; *failed is set when a wait inside a kernel gave up.
cudaError_t launch_gram(const GramPlan& g, const float* F, int N, int P, const double* mu, double* up, double* down, uint8_t* digits, double* part,
                        int* failed, cudaStream_t stream);

}  // namespace rocket
