// Ridge regressor on the pooled features (Section 3, step (3); Section 3.3): fit and predict on the
// device, so that features never have to leave it.
//
// Fit, with an intercept that is not penalised: centre the columns of F [N][P] and y, solve the dual
// system (Fc Fc^T + alpha I) a = yc (N x N, N examples << P features), w = Fc^T a,
// b = mean(y) - mean(F) . w.  The Gram matrix (of larger problems by rocket_gram.cu), its Cholesky factor and the two triangular solves are
// kept in double precision: the features are fp32 data, everything derived from them is not rounded
// to fp32 before w and b are stored.  Every sum is taken in an order that depends on the sizes alone, so two fits
// of the same data are bitwise identical.
//
// Measured at 677 x 20,000 (B200): column means, Gram matrix, factorisation with solves and weights take
// 18 / 193 (in FP64 496) / 381 / 21 us; as one thread per column, 2 x 2 outputs per thread, one block and one thread per column they took
// 55 / 2,607 / 20,270 / 174.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "rocket_gram.h"
#include "rocket_internal.h"

namespace rocket {
namespace {

namespace cg = cooperative_groups;

constexpr int kRThreads = 256;
constexpr int kRWarps = kRThreads / 32;

// Column kernels: a block owns 32 columns (a lane each, so that a warp reads 128 contiguous bytes of a row) and its
// eight warps share the rows; the warps' sums are added in warp order.
//
// mu[p] = mean over the N rows of F[.][p]; the block past the last column takes ybar = mean(y) and clears the ticket
// the weights kernel counts its blocks with and the flag of waits that gave up.
__global__ void __launch_bounds__(kRThreads)
ridge_means_kernel(const float* __restrict__ F, const float* __restrict__ y, int N, int P, double* __restrict__ mu,
                   double* __restrict__ ybar, unsigned* __restrict__ ticket, int* __restrict__ failed) {
    __shared__ double red[kRWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool targets = (int)blockIdx.x * 32 >= P;
    const int p = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (targets) {
        for (int i = threadIdx.x; i < N; i += kRThreads) s += (double)y[i];
    } else if (p < P) {
        const float* __restrict__ f = F + p;
#pragma unroll 8
        for (int i = warp; i < N; i += kRWarps) s += (double)__ldg(f + (size_t)i * P);
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int w = 1; w < kRWarps; ++w) s += red[w][lane];
        if (targets) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) { *ybar = s / (double)N; *ticket = 0u; *failed = 0; }
        } else if (p < P) {
            mu[p] = s / (double)N;
        }
    }
}

// One 64 x 64 tile of the lower triangle of G over a slice of the feature axis, as a partial sum.  Bound: the FP64 rate
// (64 multiply-adds per clock and SM, reached by the FP64 matrix instruction with eight warps per SM; the scalar form
// reaches 58.7 and loads twelve shared-memory words for 32 products where the fragments below take eight for 128).  A
// warp owns 32 x 32 outputs as 4 x 4 fragments of m8n8k4; the slice goes through shared memory 32 columns at a time,
// centred on the way in, the next piece on its way in registers.  A row of the staged piece is 36 doubles, so that the
// 16 lanes of a fragment load's half warp (4 rows x 4 columns) fall on 16 different bank pairs.
constexpr int kGT = 64, kGP = 32, kGPitch = kGP + 4, kGThreads = 128;
constexpr int kGRows = 2 * kGT * kGP / kGThreads;      // staged values per thread and piece (half of them of each operand)
__global__ void __launch_bounds__(kGThreads, 4)
ridge_gram_kernel(const float* __restrict__ F, int N, int P, const double* __restrict__ mu, int slice,
                  double* __restrict__ part) {
    extern __shared__ double smem[];
    double (*A)[kGPitch] = reinterpret_cast<double (*)[kGPitch]>(smem);
    double (*B)[kGPitch] = A + kGT;
    // tile index -> (bi, bj) with bj <= bi
    int bi = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
    while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
    while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
    const int bj = blockIdx.x - bi * (bi + 1) / 2;
    const int p_beg = blockIdx.y * slice, p_end = min(P, p_beg + slice);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = lane, row0 = warp;                      // staging: thread takes column `col` of rows row0 + 4 i
    const int wr = (warp >> 1) * 32, wc = (warp & 1) * 32;  // the warp's outputs
    const int fr = lane >> 2, fk = lane & 3;
    double acc[4][4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v][0] = acc[u][v][1] = 0.0;
    float x[kGRows];
    double m = 0.0;
    auto fetch = [&](int p0) {
        const int p = p0 + col;
        const bool ok = p < p_end;
        m = ok ? mu[p] : 0.0;
#pragma unroll
        for (int i = 0; i < kGRows / 2; ++i) {
            const int ra = bi * kGT + row0 + 4 * i, rb = bj * kGT + row0 + 4 * i;
            x[i] = ok && ra < N ? __ldg(F + (size_t)ra * P + p) : 0.0f;
            x[kGRows / 2 + i] = ok && rb < N ? __ldg(F + (size_t)rb * P + p) : 0.0f;
        }
    };
    fetch(p_beg);
    for (int p0 = p_beg; p0 < p_end; p0 += kGP) {
        __syncthreads();
        const bool ok = p0 + col < p_end;
#pragma unroll
        for (int i = 0; i < kGRows / 2; ++i) {
            const int r = row0 + 4 * i;
            A[r][col] = ok && bi * kGT + r < N ? (double)x[i] - m : 0.0;
            B[r][col] = ok && bj * kGT + r < N ? (double)x[kGRows / 2 + i] - m : 0.0;
        }
        __syncthreads();
        if (p0 + kGP < p_end) fetch(p0 + kGP);
#pragma unroll
        for (int k = 0; k < kGP; k += 4) {
            double a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = A[wr + 8 * u + fr][k + fk];
                b[u] = B[wc + 8 * u + fr][k + fk];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                                 : "+d"(acc[u][v][0]), "+d"(acc[u][v][1]) : "d"(a[u]), "d"(b[v]));
        }
    }
    double* __restrict__ out = part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (kGT * kGT);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
            *reinterpret_cast<double2*>(out + (wr + 8 * u + fr) * kGT + wc + 8 * v + 2 * fk) =
                make_double2(acc[u][v][0], acc[u][v][1]);
}

// ---- Cholesky factor and solves -------------------------------------------------------------------------------
// G [Np][Np] (Np a multiple of 32 above N) holds the lower triangle of Fc Fc^T + alpha I, row N holds yc^T, rows below are
// zero: the factorisation then leaves z = L^-1 yc in row N by itself.  Blocks of 32 x 32, right-looking: at step kb every
// block of the grid factors the diagonal block for itself (one warp, a row per lane), solves the two panel blocks its
// tile needs and updates the tile, so that a step takes one grid-wide barrier and no panel travels between barriers.
// Solved panel blocks go transposed into the upper triangle, diagonal factors into Ld.  Bound: the chain of steps (22 of
// them at N = 677; a diagonal block is 32 dependent pivots), not arithmetic.
constexpr int kCB = 32, kCThreads = 256, kCPitch = kCB + 1, kDPitch = kCB + 2;

struct CholArgs {
    const double* part;       // partial Gram tiles [slices][tiles][64][64]
    int slices, tiles;
    double alpha;
    const float* y;
    const double* ybar;
    double* G;
    double* Ld;               // diagonal factors [nb][32][32]
    double* a;                // solution [N]
    int* status;              // 0 = ok, 1 = a pivot was not positive
    int N, Np;
};

// Factors the leading `ncols` columns of the block whose rows are held by the lanes (s[lane][0 .. lane]); the factor's
// transpose goes to t (t[j][c] = L[c][j]), the reciprocal pivots to rinv.  One warp.
__device__ __forceinline__ bool chol_factor_block(const double (*s)[kCPitch], double (*t)[kDPitch], double* rinv, int ncols,
                                                  int lane) {
    double a[kCB];
    bool good = true;
#pragma unroll
    for (int c = 0; c < kCB; ++c) a[c] = s[lane][c];
#pragma unroll
    for (int j = 0; j < kCB; ++j) {
        if (j < ncols) {
            double d = __shfl_sync(0xffffffffu, a[j], j);
            if (!(d > 0.0)) { good = false; d = 1.0; }
            const double r = rsqrt(d);
            const double l = lane == j ? d * r : a[j] * r;
            t[j][lane] = lane >= j ? l : 0.0;
            if (lane == 0) rinv[j] = r;
            __syncwarp();
#pragma unroll
            for (int c = j + 1; c < kCB; ++c) a[c] -= l * t[j][c];
        }
    }
    __syncwarp();
    return good;
}

// Row `lane` of a panel block: x L^T = g, in place.  One warp.
__device__ __forceinline__ void chol_solve_row(double (*p)[kCPitch], const double (*t)[kDPitch], const double* rinv, int lane) {
    double g[kCB];
#pragma unroll
    for (int c = 0; c < kCB; ++c) g[c] = p[lane][c];
#pragma unroll
    for (int j = 0; j < kCB; ++j) {
        const double x = g[j] * rinv[j];
        g[j] = x;
#pragma unroll
        for (int c = j + 1; c < kCB; ++c) g[c] -= x * t[j][c];
    }
#pragma unroll
    for (int c = 0; c < kCB; ++c) p[lane][c] = g[c];
}

__global__ void __launch_bounds__(kCThreads)
ridge_cholesky_solve_kernel(CholArgs q) {
    __shared__ double s_t[kCB][kDPitch];
    __shared__ double s_rinv[kCB];
    __shared__ double s_raw[ROCKET_RIDGE_MAX_EXAMPLES];      // the panel blocks; in the end the solution
    static_assert(2 * kCB * kCPitch <= ROCKET_RIDGE_MAX_EXAMPLES, "two panel blocks fit");
    double (*s_pi)[kCPitch] = reinterpret_cast<double (*)[kCPitch]>(s_raw);
    double (*s_pj)[kCPitch] = s_pi + kCB;
    cg::grid_group grid = cg::this_grid();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = q.N, Np = q.Np, nb = Np / kCB;
    double* __restrict__ G = q.G;

    // lower blocks of G from the partial tiles, in slice order
    const int blocks = nb * (nb + 1) / 2;
    for (int b = blockIdx.x; b < blocks; b += gridDim.x) {
        int ib = (int)((sqrtf(8.0f * (float)b + 1.0f) - 1.0f) * 0.5f);
        while (ib * (ib + 1) / 2 > b) --ib;
        while ((ib + 1) * (ib + 2) / 2 <= b) ++ib;
        const int jb = b - ib * (ib + 1) / 2;
        for (int e = tid; e < kCB * kCB; e += kCThreads) {
            const int i = ib * kCB + e / kCB, j = jb * kCB + e % kCB;
            double g = 0.0;
            if (i < N && j < N) {
                const int ti = i / kGT, tj = j / kGT;
                const double* __restrict__ src = q.part + (size_t)(ti * (ti + 1) / 2 + tj) * (kGT * kGT) + (i % kGT) * kGT + j % kGT;
#pragma unroll 4
                for (int v = 0; v < q.slices; ++v) g += src[(size_t)v * q.tiles * (kGT * kGT)];
                if (i == j) g += q.alpha;
            } else if (i == N && j < N) {
                g = (double)q.y[j] - *q.ybar;
            }
            G[(size_t)i * Np + j] = g;
        }
    }
    if (blockIdx.x == 0 && tid == 0) *q.status = 0;
    grid.sync();

    bool good = true;
    for (int kb = 0; kb < nb; ++kb) {
        const int k0 = kb * kCB, ncols = min(kCB, N - k0);
        const int rest = nb - kb - 1, tiles = rest * (rest + 1) / 2;
        if (ncols > 0 && ((int)blockIdx.x < tiles || blockIdx.x == 0)) {
            for (int e = tid; e < kCB * kCB; e += kCThreads) s_pi[e / kCB][e % kCB] = G[(size_t)(k0 + e / kCB) * Np + k0 + e % kCB];
            __syncthreads();
            if (warp == 0) good = chol_factor_block(s_pi, s_t, s_rinv, ncols, lane) && good;
            __syncthreads();
            if (blockIdx.x == 0)
                for (int e = tid; e < kCB * kCB; e += kCThreads)
                    q.Ld[(size_t)kb * kCB * kCB + e] = s_t[e % kCB][e / kCB];    // Ld[r][c] = L[r][c], read below r's diagonal only
            for (int b = blockIdx.x; b < tiles; b += gridDim.x) {
                // tile (ib, jb) of the trailing blocks, column by column so that the first ones are the panel's own
                int x = (int)((sqrtf(8.0f * (float)(tiles - 1 - b) + 1.0f) - 1.0f) * 0.5f);
                while (x * (x + 1) / 2 > tiles - 1 - b) --x;
                while ((x + 1) * (x + 2) / 2 <= tiles - 1 - b) ++x;
                const int jb = nb - 1 - x, ib = nb - 1 - ((tiles - 1 - b) - x * (x + 1) / 2);
                const int i0 = ib * kCB, j0 = jb * kCB;
                for (int e = tid; e < kCB * kCB; e += kCThreads) {
                    const int r = e / kCB, c = e % kCB;
                    s_pi[r][c] = G[(size_t)(i0 + r) * Np + k0 + c];
                    if (ib != jb) s_pj[r][c] = G[(size_t)(j0 + r) * Np + k0 + c];
                }
                const int ty = tid / 16, tx = tid % 16;
                double g[2][2];
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) g[u][v] = G[(size_t)(i0 + ty + 16 * u) * Np + j0 + tx + 16 * v];
                __syncthreads();
                if (warp == 0) chol_solve_row(s_pi, s_t, s_rinv, lane);
                else if (warp == 1 && ib != jb) chol_solve_row(s_pj, s_t, s_rinv, lane);
                __syncthreads();
                const double (*pj)[kCPitch] = ib != jb ? s_pj : s_pi;
#pragma unroll 8
                for (int k = 0; k < kCB; ++k) {
                    const double a0 = s_pi[ty][k], a1 = s_pi[ty + 16][k], b0 = pj[tx][k], b1 = pj[tx + 16][k];
                    g[0][0] -= a0 * b0; g[0][1] -= a0 * b1; g[1][0] -= a1 * b0; g[1][1] -= a1 * b1;
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) G[(size_t)(i0 + ty + 16 * u) * Np + j0 + tx + 16 * v] = g[u][v];
                if (jb == kb + 1)
                    for (int e = tid; e < kCB * kCB; e += kCThreads) G[(size_t)(k0 + e / kCB) * Np + i0 + e % kCB] = s_pi[e % kCB][e / kCB];
                __syncthreads();
            }
        }
        if (rest > 0) grid.sync();
    }
    if (blockIdx.x != 0) return;

    // L^T a = z, from the last block up.  Row k0 + j of the upper triangle holds L's column: a warp per row takes the
    // part below the diagonal block, one warp solves the diagonal block.
    if (warp == 0 && lane == 0 && !good) *q.status = 1;
    __syncthreads();
    double* s_a = s_raw;
    const int nblk = (N + kCB - 1) / kCB;
    for (int kb = nblk - 1; kb >= 0; --kb) {
        const int k0 = kb * kCB, ncols = min(kCB, N - k0);
        for (int e = tid; e < kCB * kCB; e += kCThreads) s_t[e / kCB][e % kCB] = q.Ld[(size_t)kb * kCB * kCB + e];   // s_t[r][c] = L[r][c]
        double sum[kCB / (kCThreads / 32)];
#pragma unroll
        for (int u = 0; u < kCB / (kCThreads / 32); ++u) sum[u] = 0.0;
        for (int i = k0 + kCB + lane; i < N; i += 32) {
            const double ai = s_a[i];
#pragma unroll
            for (int u = 0; u < kCB / (kCThreads / 32); ++u)
                sum[u] += G[(size_t)(k0 + warp + (kCThreads / 32) * u) * Np + i] * ai;
        }
#pragma unroll
        for (int u = 0; u < kCB / (kCThreads / 32); ++u) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
            if (lane == 0) s_rinv[warp + (kCThreads / 32) * u] = sum[u];
        }
        __syncthreads();
        if (warp == 0) {
            double z = 0.0;
            if (lane < ncols) z = (N / kCB == kb ? q.Ld[(size_t)kb * kCB * kCB + (N - k0) * kCB + lane] : G[(size_t)(k0 + lane) * Np + N]);
            double v = lane < ncols ? z - s_rinv[lane] : 0.0;
            const double inv = lane < ncols ? 1.0 / s_t[lane][lane] : 0.0;
#pragma unroll 4
            for (int j = ncols - 1; j >= 0; --j) {
                const double aj = __shfl_sync(0xffffffffu, v * inv, j);
                if (lane == j) v = aj;
                else if (lane < j) v -= s_t[j][lane] * aj;
            }
            if (lane < ncols) { s_a[k0 + lane] = v; q.a[k0 + lane] = v; }
        }
        __syncthreads();
    }
}

// w[p] = sum_i a[i] (F[i][p] - mu[p]), and the intercept b = ybar - sum_p mu[p] w[p] (with the stored fp32 weights) by the
// last block to finish, in block order.
__global__ void __launch_bounds__(kRThreads)
ridge_weights_kernel(const float* __restrict__ F, int N, int P, const double* __restrict__ mu, const double* __restrict__ a,
                     const double* __restrict__ ybar, float* __restrict__ w, float* __restrict__ b, double* __restrict__ part,
                     unsigned* __restrict__ ticket) {
    __shared__ double s_a[ROCKET_RIDGE_MAX_EXAMPLES];
    __shared__ double red[kRWarps][32];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < N; i += kRThreads) s_a[i] = a[i];
    __syncthreads();
    const int p = blockIdx.x * 32 + lane;
    double s = 0.0, m = 0.0;
    if (p < P) {
        m = mu[p];
        const float* __restrict__ f = F + p;
#pragma unroll 8
        for (int i = warp; i < N; i += kRWarps) s += s_a[i] * ((double)__ldg(f + (size_t)i * P) - m);
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int v = 1; v < kRWarps; ++v) s += red[v][lane];
        if (p < P) w[p] = (float)s;
        double c = p < P ? m * (double)(float)s : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0) {
            part[blockIdx.x] = c;
            __threadfence();
            s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double c = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kRThreads) c += __ldcg(part + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) red[warp][0] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < kRWarps; ++v) c += red[v][0];
        *b = (float)(*ybar - c);
    }
}

// yhat[n] = b + sum_p F[n][p] w[p], products summed in double: a row per block of 256 threads (W = 8 warps), half a
// block or a warp.  (Eight loads of a lane gathered in registers before the first product: 68 us for 4,000 rows of 20,000 against 64.)
template <bool VEC, int W>
__global__ void __launch_bounds__(kRThreads)
ridge_predict_rows_kernel(const float* __restrict__ F, int N, int P, const float* __restrict__ w, const float* __restrict__ b,
                          float* __restrict__ yhat) {
    __shared__ double red[kRWarps];
    const int warp = threadIdx.x >> 5, at = threadIdx.x % (32 * W);
    const long long n = (long long)blockIdx.x * (kRWarps / W) + warp / W;
    double s = 0.0;
    if (n < N) {
        const float* __restrict__ f = F + (size_t)n * P;
        if (VEC) {
            const float4* __restrict__ f4 = reinterpret_cast<const float4*>(f);
            const float4* __restrict__ w4 = reinterpret_cast<const float4*>(w);
            const int n4 = P / 4;
#pragma unroll 4
            for (int i = at; i < n4; i += 32 * W) {
                const float4 x = __ldg(f4 + i), v = __ldg(w4 + i);
                s += (double)x.x * (double)v.x + (double)x.y * (double)v.y + ((double)x.z * (double)v.z + (double)x.w * (double)v.w);
            }
        } else {
#pragma unroll 4
            for (int i = at; i < P; i += 32 * W) s += (double)__ldg(f + i) * (double)__ldg(w + i);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (W > 1) {
        if ((threadIdx.x & 31) == 0) red[warp] = s;
        __syncthreads();
        if (at == 0)
            for (int v = 1; v < W; ++v) s += red[warp + v];
    }
    if (n < N && at == 0) yhat[n] = (float)(s + (double)*b);
}

// The same for few, long rows: the blocks of a cluster (as many as it takes to put two blocks on every SM, at most eight) share a
// row, each sums its contiguous part, the first adds the parts in rank order through distributed shared memory.  Bound: the
// latency of a few trips to memory: 60 rows of 20,000 take 3.7 us on the device, 5.8 with a block per row.
constexpr int kPThreads = 512;
constexpr int kPPairs = 148;                            // rows that two blocks each share: two blocks per SM of this GPU
template <bool VEC>
__global__ void __launch_bounds__(kPThreads)
ridge_predict_kernel(const float* __restrict__ F, int P, const float* __restrict__ w, const float* __restrict__ b,
                     float* __restrict__ yhat) {
    __shared__ double red[kPThreads / 32];
    __shared__ double s_part[8];
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = gridDim.x, rank = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // No block may write to the first one's shared memory before that block runs: every block says here that it does, and waits for
    // the others behind its loop.
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const float* __restrict__ f = F + (size_t)blockIdx.y * P;
    double s = 0.0;
    if (VEC) {
        const int n4 = P / 4, beg = (int)((long long)n4 * rank / parts), end = (int)((long long)n4 * (rank + 1) / parts);
        const float4* __restrict__ f4 = reinterpret_cast<const float4*>(f);
        const float4* __restrict__ w4 = reinterpret_cast<const float4*>(w);
#pragma unroll 4
        for (int i = beg + threadIdx.x; i < end; i += kPThreads) {
            const float4 x = __ldg(f4 + i), v = __ldg(w4 + i);
            s += (double)x.x * (double)v.x + (double)x.y * (double)v.y + ((double)x.z * (double)v.z + (double)x.w * (double)v.w);
        }
    } else {
        const int beg = (int)((long long)P * rank / parts), end = (int)((long long)P * (rank + 1) / parts);
#pragma unroll 8
        for (int i = beg + threadIdx.x; i < end; i += kPThreads) s += (double)__ldg(f + i) * (double)__ldg(w + i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
        s = lane < kPThreads / 32 ? red[lane] : 0.0;
#pragma unroll
        for (int o = kPThreads / 64; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *cluster.map_shared_rank(&s_part[rank], 0) = s;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
        s = s_part[0];
        for (int r = 1; r < parts; ++r) s += s_part[r];
        yhat[blockIdx.y] = (float)(s + (double)*b);
    }
}

int status_of(cudaError_t e) {
    if (e == cudaSuccess) return ROCKET_OK;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? ROCKET_ENOMEM : ROCKET_ECUDA;
}

// Workspace of a fit.  cudaMalloc and cudaFree take 0.4 to 5 ms each here, several times the fit itself, so one buffer
// per device, of at most kKeepBytes, outlives the call: a fit takes it while nobody else has it and puts it back after its
// stream has finished; a larger or a concurrent fit allocates and frees its own.  The buffer is given back when a handle
// of the library is destroyed and when a device allocation of the library fails (release_cached_workspaces).
constexpr size_t kKeepBytes = (size_t)128 << 20;
constexpr int kMaxDevices = 64;
struct Kept { void* ptr = nullptr; size_t bytes = 0; bool taken = false; };
std::mutex g_kept_mu;
Kept g_kept[kMaxDevices];

struct FitWorkspace {
    void* ptr = nullptr;
    int slot = -1;          // >= 0: the device's kept buffer
    cudaError_t take(size_t bytes) {
        int dev = -1;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (bytes <= kKeepBytes && dev < kMaxDevices) {
            std::lock_guard<std::mutex> lk(g_kept_mu);
            Kept& k = g_kept[dev];
            if (!k.taken && k.bytes >= bytes) {
                k.taken = true;
                slot = dev;
                ptr = k.ptr;
                return cudaSuccess;
            }
        }
        return device_malloc(&ptr, bytes);
    }
    // the work that used it has finished
    void put_back(size_t bytes) {
        void* gone = ptr;
        int dev = -1;
        if (slot >= 0) {
            std::lock_guard<std::mutex> lk(g_kept_mu);
            g_kept[slot].taken = false;
            return;
        }
        if (bytes <= kKeepBytes && cudaGetDevice(&dev) == cudaSuccess && dev < kMaxDevices) {
            std::lock_guard<std::mutex> lk(g_kept_mu);
            Kept& k = g_kept[dev];
            if (!k.taken && k.bytes < bytes) {       // the larger buffer stays
                gone = k.ptr;
                k.ptr = ptr;
                k.bytes = bytes;
            }
        }
        if (gone) cudaFree(gone);
    }
};

}  // namespace

void release_cached_workspaces() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev >= kMaxDevices) { cudaGetLastError(); return; }
    void* gone = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_kept_mu);
        Kept& k = g_kept[dev];
        if (!k.taken) { gone = k.ptr; k = Kept(); }
    }
    if (gone) cudaFree(gone);
}

}  // namespace rocket

using namespace rocket;

extern "C" int rocket_ridge_fit(const float* feat_dev, int N, int P, const float* y_dev, float alpha, float* w_dev,
                                float* b_dev, void* cuda_stream) {
    if (!feat_dev || !y_dev || !w_dev || !b_dev || N < 1 || P < 1) return ROCKET_EINVAL;
    if (!(alpha >= 0.0f) || !(alpha < 3.0e38f)) return ROCKET_EINVAL;
    if (N > ROCKET_RIDGE_MAX_EXAMPLES) return ROCKET_EUNSUPPORTED;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t gram_smem = (size_t)2 * kGT * kGPitch * sizeof(double);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ridge_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gram_smem);
    if (e != cudaSuccess) return status_of(e);
    const int col_blocks = (P + 31) / 32;
    // Slices of the feature axis: about two waves of the four blocks an SM holds, at least 128 columns each, and no more
    // than 40 MB of partial tiles (or one slice, 65 MB at the most examples).
    const int nt = (N + kGT - 1) / kGT, tiles = nt * (nt + 1) / 2;
    const size_t tile_bytes = (size_t)kGT * kGT * sizeof(double);
    // Integers on the tensor cores from about 100 examples of 20,000 features on (us, FP64 and integers: 24 x 20,000 99 and 113, 97 x 3,001
    // 111 and 121, 300 x 600 207 and 212, 100 x 20,000 166 and 155, 300 x 5,000 238 and 225, 677 x 20,000 931 and 632).
    const bool integers = (double)N * N * P >= 1.2e8;
    const GramPlan gram = gram_plan(N, P, sms);
    int slices = std::max(1, std::min({8 * sms / tiles, P / 128, (int)(((size_t)40 << 20) / (tile_bytes * tiles))}));
    const int slice = ((P + slices - 1) / slices + kGP - 1) / kGP * kGP;
    slices = integers ? gram.slices : (P + slice - 1) / slice;
    const int nb = (N + 1 + kCB - 1) / kCB, Np = nb * kCB;
    // workspace: mu[P], a[N], part[col_blocks], ybar, G[Np][Np], Ld[nb][32][32], partial Gram tiles, ticket, status
    size_t off = 0;
    auto take = [&](size_t doubles) { const size_t o = off; off += (doubles + 31) / 32 * 32; return o; };
    const size_t o_mu = take(P), o_a = take(N), o_part = take(col_blocks), o_ybar = take(1), o_G = take((size_t)Np * Np);
    const size_t o_Ld = take((size_t)nb * kCB * kCB), o_gram = take((size_t)slices * tiles * kGT * kGT), o_int = take(2);
    const size_t o_up = take(integers ? N : 0), o_down = take(integers ? N : 0), o_digits = take(integers ? gram.digit_bytes / sizeof(double) : 0);
    const size_t bytes = off * sizeof(double);
    FitWorkspace ws;
    if ((e = ws.take(bytes)) != cudaSuccess) return status_of(e);
    double* d = static_cast<double*>(ws.ptr);
    unsigned* ticket = reinterpret_cast<unsigned*>(d + o_int);
    int* status = reinterpret_cast<int*>(d + o_int + 1);
    ridge_means_kernel<<<col_blocks + 1, kRThreads, 0, stream>>>(feat_dev, y_dev, N, P, d + o_mu, d + o_ybar, ticket, status + 1);
    if (integers)
        e = launch_gram(gram, feat_dev, N, P, d + o_mu, d + o_up, d + o_down, reinterpret_cast<uint8_t*>(d + o_digits), d + o_gram, status + 1, stream);
    else
        ridge_gram_kernel<<<dim3(tiles, slices), kGThreads, gram_smem, stream>>>(feat_dev, N, P, d + o_mu, slice, d + o_gram);
    CholArgs q{d + o_gram, slices, tiles, (double)alpha, y_dev, d + o_ybar, d + o_G, d + o_Ld, d + o_a, status, N, Np};
    void* args[] = {&q};
    // one block per SM: more would lengthen the grid barriers without shortening the chain
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(ridge_cholesky_solve_kernel),
                                    dim3((unsigned)std::max(1, std::min(sms, nb * (nb + 1) / 2))), dim3(kCThreads), args, 0, stream);
    ridge_weights_kernel<<<col_blocks, kRThreads, 0, stream>>>(feat_dev, N, P, d + o_mu, d + o_a, d + o_ybar, w_dev, b_dev,
                                                               d + o_part, ticket);
    count_launch(4);
    int host_status[2] = {0, 0};
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(host_status, status, sizeof(host_status), cudaMemcpyDeviceToHost, stream);
    const cudaError_t done = cudaStreamSynchronize(stream);
    ws.put_back(bytes);
    if (e == cudaSuccess) e = done;
    if (e != cudaSuccess) return status_of(e);
    if (host_status[1] != 0) return ROCKET_ECUDA;
    return host_status[0] == 0 ? ROCKET_OK : ROCKET_EINVAL;
}

extern "C" int rocket_ridge_predict(const float* feat_dev, int N, int P, const float* w_dev, const float* b_dev,
                                    float* yhat_dev, void* cuda_stream) {
    if (N < 0 || P < 1) return ROCKET_EINVAL;
    if (N == 0) return ROCKET_OK;
    if (!feat_dev || !w_dev || !b_dev || !yhat_dev) return ROCKET_EINVAL;
    const bool vec = P % 4 == 0 && ((reinterpret_cast<uintptr_t>(feat_dev) | reinterpret_cast<uintptr_t>(w_dev)) & 15u) == 0;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // A cluster per row where two blocks per row leave no SM with more than two, and a part is at least three loads per thread: 10 rows
    // of 20,000 take 3.1 us so and 5.6 with a block per row, 60 of 8,000 3.3 and 3.7; rows of 4,096 2.8 and 2.3.
    if (N <= kPPairs && P >= 6144) {
        unsigned parts = 2;
        while (parts < 8 && (int)parts * N <= kPPairs && (int)parts * 2 * kPThreads * 4 <= P) parts *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(parts, (unsigned)N);
        cfg.blockDim = dim3(kPThreads);
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = parts;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const cudaError_t e = vec ? cudaLaunchKernelEx(&cfg, ridge_predict_kernel<true>, feat_dev, P, w_dev, b_dev, yhat_dev)
                                  : cudaLaunchKernelEx(&cfg, ridge_predict_kernel<false>, feat_dev, P, w_dev, b_dev, yhat_dev);
        count_launch();
        return status_of(e);
    }
    // A warp per row where a lane's loads are one, or few for the number of rows (30,000 rows of 200: 6.7 us, of 2,000: 55; a block
    // per row takes 28 and 65, a cluster of one block 128 and 167; 700 rows of 600: 2.8 us so, 2.2 with a block per row).  Half a
    // block for the longer of many rows (4,000 rows of 20,000: 60 us against 64, of 4,096 the same).
    const long long loads = ((long long)P / (vec ? 4 : 1) + 31) / 32;
    auto launch = [&](auto kernel, int rows) {
        kernel<<<(unsigned)(((long long)N + rows - 1) / rows), kRThreads, 0, stream>>>(feat_dev, N, P, w_dev, b_dev, yhat_dev);
    };
    if (loads <= 1 || N >= 300 * loads) vec ? launch(ridge_predict_rows_kernel<true, 1>, 8) : launch(ridge_predict_rows_kernel<false, 1>, 8);
    else if (N >= 2000) vec ? launch(ridge_predict_rows_kernel<true, 4>, 2) : launch(ridge_predict_rows_kernel<false, 4>, 2);
    else vec ? launch(ridge_predict_rows_kernel<true, 8>, 1) : launch(ridge_predict_rows_kernel<false, 8>, 1);
    count_launch();
    return status_of(cudaGetLastError());
}
