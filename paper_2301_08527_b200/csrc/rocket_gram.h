// Gram matrix of the centred features in integers on the tensor cores (rocket_gram.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace rocket {

constexpr size_t kGramDigitBytes = (size_t)112 << 20;   // digits of as many columns at a time

struct GramPlan {
    int groups, blocks_mn;     // groups of 8 rows; 128 x 64 tiles of the lower triangle
    int chunk, slices;         // blocks of 64 columns whose digits are held at a time; slices of partial tiles
    size_t digit_bytes;
};
GramPlan gram_plan(int N, int P, int sms);

// Partial tiles part[slices][tiles of the lower triangle, 64 x 64][64][64] of Fc Fc^T.  up, down: N doubles each; digits: digit_bytes, 128-byte
// aligned; *failed is set when a wait inside a kernel gave up.
cudaError_t launch_gram(const GramPlan& g, const float* F, int N, int P, const double* mu, double* up, double* down, uint8_t* digits, double* part,
                        int* failed, cudaStream_t stream);

}  // namespace rocket
