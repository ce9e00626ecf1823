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
// 18 / 255 (in FP64 496) / 228 (381 before) / 21 us; as one thread per column, 2 x 2 outputs per thread, one block and one thread per column they took
// 55 / 2,607 / 20,270 / 174.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "rocket_gram.h"
#include "rocket_internal.h"
#include "rocket_pivot.cuh"

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
// zero: the factorisation then leaves z = L^-1 yc in row N by itself.  Blocks of 32 x 32, right-looking, one grid-wide barrier per
// step: block 0 updates the next diagonal block first and factors it while the others update the rest, and what it passes on is the
// factor and its inverse, so that the panel blocks a tile needs are products that 256 threads share.  Solved panel blocks go transposed
// into the upper triangle, factors and inverses into Li and Mi.  Bound: block 0's chain of 32 dependent pivots per step (22 steps at N = 677).
//
// A product with an explicit inverse is off by 2^-53 times the condition of the diagonal block, where a substitution is off by 2^-53 of its own
// terms: X = A M alone left rows of 10^-4 to 10^4 with errors 10 to 400 times as large, or refused them for a pivot that was not positive.  So
// where the factor or its inverse has an element far beyond the others (kCLarge) a product takes one step of iterative refinement,
// X + (A - X L^T) M, which leaves the square of that error: the same as a substitution's up to conditions of 10^8 of a factor, which is as far
// as any factorisation in double precision goes.  In every block it takes 26 us at 677 x 20,000; left out where no element is beyond 2, 8 or 32
// times the others, the errors of sixty fits of twelve kinds were the same to three digits.  It takes 1 us where no block does.
constexpr int kCB = 32, kCThreads = 256, kCPitch = kCB + 4, kDPitch = kCB + 2;
constexpr double kCLarge = 8.0;                                       // times the largest diagonal of the factor or the least of its inverse
constexpr int kCSmem = kCB * kDPitch + 6 * kCB * kCPitch;              // doubles: a factor and six blocks; in the end the solution besides

struct CholArgs {
    const double* part;       // partial Gram tiles [slices][tiles][64][64]
    int slices, tiles;
    double alpha;
    const float* y;
    const double* ybar;
    double* G;
    double* Mi;               // inverse factors of the diagonal blocks, transposed [nb][32][32]
    double* Li;               // the factors, transposed [nb][32][32]
    int* refine;              // whether products with the inverse take a refinement step [nb]
    double* z;                // row N of the factor, by blocks
    double* a;                // solution [N]
    int* status;              // 0 = ok, 1 = a pivot was not positive
    int N, Np;
};

// Factors the leading `ncols` columns of the block whose rows are held by the lanes (s[lane][0 .. lane]) and inverts the factor: row r
// of the inverse's transpose goes to m[r]; lane j returns in root the reciprocal of the factor's diagonal j, which is in t[j][32] as well (their
// least in t[0][33]), and t[j] holds column j of the factor times that diagonal.  One warp.
//
// A double-precision operation takes some 40 clocks here, so what counts is how many of them lie between a pivot and the next.  The
// elimination is square-root free (a_ik -= c_ij c_kj / d_j with unscaled columns c), 1 / d_j is y (1 + p) with a p that is ready one operation after y
// (pivot_reciprocal), and the next pivot's column takes a - g - g p with g = c_ij c_kj y ready by then: three operations after the approximation.
// With the factor's own columns and 1 / sqrt(d_j) they were six: 10,800 clocks for a block, 8,400 now.  (One body for all pivots, the rows
// moving down by a column each time, has twice the multiply-adds: 13,700.)
__device__ __forceinline__ bool chol_factor_block(const double (*s)[kCPitch], double (*t)[kDPitch], double (*m)[kCPitch], int ncols, int lane, double& root) {
    double a[kCB], x[kCB], mine = 1.0;
    bool good = true;
#pragma unroll
    for (int c = 0; c < kCB; ++c) {
        a[c] = s[lane][c];
        x[c] = c == lane ? 1.0 : 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kCB; ++j) {
        const bool there = j < ncols;
        double d = __shfl_sync(0xffffffffu, a[j], j), y, p;
        good = good && (!there || d >= 2.2250738585072014e-308);
        d = there && d >= 2.2250738585072014e-308 ? d : 1.0;
        pivot_reciprocal(d, y, p);
        const double col = there && lane >= j ? a[j] : 0.0;
        if (lane == j) mine = d;
        t[j][lane] = col;
        const double cy = col * y;
        if (j + 1 < kCB) {                             // what the next pivot waits for
            const double next = __shfl_sync(0xffffffffu, col, j + 1), g = cy * next;
            a[j + 1] = fma(-g, p, a[j + 1] - g);
        }
        __syncwarp();
        const double f = fma(cy, p, cy), xs = there ? times_reciprocal(x[j], y, p) : 0.0;
        if (j + 1 < kCB) x[j + 1] = fma(-xs, t[j][j + 1], x[j + 1]);
#pragma unroll
        for (int c = j + 2; c < kCB; ++c) {
            const double lc = t[j][c];
            a[c] = fma(-f, lc, a[c]);
            x[c] = fma(-xs, lc, x[c]);
        }
    }
    root = rsqrt(mine);
    t[lane][kCB] = root;
    const int least = __reduce_min_sync(0xffffffffu, __double2hiint(root));   // positive: the high words are in their order
    if (lane == 0) t[0][kCB + 1] = __hiloint2double(least, 0);
#pragma unroll
    for (int c = 0; c < kCB; ++c) m[lane][c] = x[c] * __shfl_sync(0xffffffffu, root, c);
    __syncwarp();
    return good;
}

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

__global__ void __launch_bounds__(kCThreads)
ridge_cholesky_solve_kernel(CholArgs q) {
    extern __shared__ double smem[];
    double (*s_t)[kDPitch] = reinterpret_cast<double (*)[kDPitch]>(smem);
    double (*s_m)[kCPitch] = reinterpret_cast<double (*)[kCPitch]>(smem + kCB * kDPitch), (*s_pi)[kCPitch] = s_m + kCB, (*s_pj)[kCPitch] = s_pi + kCB;
    double (*s_l)[kCPitch] = s_pj + kCB, (*s_xi)[kCPitch] = s_l + kCB, (*s_xj)[kCPitch] = s_xi + kCB;
    cg::grid_group grid = cg::this_grid();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = q.N, Np = q.Np, nb = Np / kCB;
    // a warp's two 8 x 8 fragments of a block: those columns of a triangular factor that have as many products together for every warp
    const int fr = lane >> 2, fk = lane & 3, br = warp >> 1, bc[2] = {warp & 1, 3 - (warp & 1)};
    double* __restrict__ G = q.G;
    bool good = true;

    // the factor of diagonal block kb, whose elements are in s_pi, and its inverse (block 0)
    auto factor = [&](int kb) {
        const int ncols = min(kCB, N - kb * kCB);
        double root = 0.0;
        bool large = false;
        if (ncols > 0 && warp == 0) good = chol_factor_block(s_pi, s_t, s_m, ncols, lane, root) && good;
        __syncthreads();
        if (ncols > 0)
            for (int e = tid; e < kCB * kCB; e += kCThreads) {
                const double m = s_m[e / kCB][e % kCB], l = s_t[e / kCB][e % kCB] * s_t[e / kCB][kCB];
                q.Mi[(size_t)kb * kCB * kCB + e] = m;
                large = large || fabs(m) > kCLarge * s_t[0][kCB + 1] || fabs(l) * s_t[0][kCB + 1] > kCLarge;
            }
        // row N of the factor: within its own diagonal block the factor's rows are not kept elsewhere
        if (kb == N / kCB && tid < ncols) q.z[kb * kCB + tid] = s_t[tid][N - kb * kCB] * root;
        large = __syncthreads_or(large);
        if (large)
            for (int e = tid; e < kCB * kCB; e += kCThreads) q.Li[(size_t)kb * kCB * kCB + e] = s_t[e / kCB][e % kCB] * s_t[e / kCB][kCB];
        if (tid == 0) q.refine[kb] = large ? 1 : 0;
        __syncthreads();
    };

    // lower blocks of G from the partial tiles, in slice order; block 0 takes the first diagonal block only, and factors it meanwhile (the
    // first run through that code takes 20,000 clocks longer than the others)
    const int blocks = nb * (nb + 1) / 2, helpers = (int)gridDim.x - 1;
    for (int b = blockIdx.x; b < (blockIdx.x == 0 && helpers > 0 ? 1 : blocks); b += max(1, helpers)) {
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
            if (b == 0) s_pi[e / kCB][e % kCB] = g;
        }
    }
    if (blockIdx.x == 0 && tid == 0) *q.status = 0;
    __syncthreads();

    // step -1 only factors the first diagonal block, so that there is one copy of that code: the first run through a second one took
    // 40,000 clocks
    for (int kb = -1; kb + 1 < nb; ++kb) {
        const int k0 = kb * kCB, rest = nb - kb - 1, tiles = rest * (rest + 1) / 2;
        // block 0 takes the next diagonal block, which is tile 0, and no other unless it is alone; the others share the rest
        const int step = gridDim.x > 1 ? (int)gridDim.x - 1 : 1;
        const int first = blockIdx.x, limit = kb < 0 ? (blockIdx.x == 0 ? 1 : 0) : blockIdx.x == 0 && gridDim.x > 1 ? 1 : tiles;
        for (int b = first; b < limit; b += step) {
            if (kb >= 0) {
                // tile (ib, jb) of the trailing blocks, column by column so that the first ones are the panel's own
                int x = (int)((sqrtf(8.0f * (float)(tiles - 1 - b) + 1.0f) - 1.0f) * 0.5f);
                while (x * (x + 1) / 2 > tiles - 1 - b) --x;
                while ((x + 1) * (x + 2) / 2 <= tiles - 1 - b) ++x;
                const int jb = nb - 1 - x, ib = nb - 1 - ((tiles - 1 - b) - x * (x + 1) / 2);
                const int i0 = ib * kCB, j0 = jb * kCB;
                const bool two = ib != jb;
                // all loads of the tile at once: inverse factor, panel blocks, the warp's fragments of the tile (rows fr of row block 8 br,
                // columns 2 fk, 2 fk + 1 of column blocks bc)
                constexpr int kEach = kCB * kCB / kCThreads;
                const bool refine = __ldcg(q.refine + kb) != 0;
                double lm[kEach], li[kEach], lj[kEach], g[2][2];
#pragma unroll
                for (int u = 0; u < kEach; ++u) {
                    const int e = tid + u * kCThreads, r = e / kCB, c = e % kCB;
                    lm[u] = __ldcg(q.Mi + (size_t)kb * kCB * kCB + e);
                    li[u] = __ldcg(G + (size_t)(i0 + r) * Np + k0 + c);
                    lj[u] = two ? __ldcg(G + (size_t)(j0 + r) * Np + k0 + c) : 0.0;
                }
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const double2 w = __ldcg(reinterpret_cast<const double2*>(G + (size_t)(i0 + 8 * br + fr) * Np + j0 + 8 * bc[v] + 2 * fk));
                    g[v][0] = w.x; g[v][1] = w.y;
                }
#pragma unroll
                for (int u = 0; u < kEach; ++u) {
                    const int e = tid + u * kCThreads, r = e / kCB, c = e % kCB;
                    s_m[r][c] = lm[u];
                    s_pi[r][c] = li[u];
                    if (two) s_pj[r][c] = lj[u];
                }
                // a matrix instruction takes long, too: two sums for every fragment
                double xi[2][2] = {}, xj[2][2] = {};
                // times an upper triangle, onto xi, xj
                auto multiply = [&](const double (*pi)[kCPitch], const double (*pj)[kCPitch], const double (*by)[kCPitch], double sign) {
                    double h0[2][2] = {}, h1[2][2] = {};
#pragma unroll
                    for (int k = 0; k < kCB; k += 4) {
                        const double x = sign * pi[8 * br + fr][k + fk], y = two ? sign * pj[8 * br + fr][k + fk] : 0.0;
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            if (k >= 8 * bc[v] + 8) continue;      // zeros
                            const double m = by[k + fk][8 * bc[v] + fr];
                            dmma(k & 4 ? h0[v] : xi[v], x, m);
                            if (two) dmma(k & 4 ? h1[v] : xj[v], y, m);
                        }
                    }
#pragma unroll
                    for (int v = 0; v < 2; ++v)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            xi[v][h] += h0[v][h];
                            xj[v][h] += h1[v][h];
                        }
                };
                auto fetch = [&](const double (*pi)[kCPitch], const double (*pj)[kCPitch]) {
#pragma unroll
                    for (int v = 0; v < 2; ++v)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            xi[v][h] = pi[8 * br + fr][8 * bc[v] + 2 * fk + h];
                            xj[v][h] = two ? pj[8 * br + fr][8 * bc[v] + 2 * fk + h] : 0.0;
                        }
                };
                auto keep = [&](double (*pi)[kCPitch], double (*pj)[kCPitch]) {
#pragma unroll
                    for (int v = 0; v < 2; ++v)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            pi[8 * br + fr][8 * bc[v] + 2 * fk + h] = xi[v][h];
                            if (two) pj[8 * br + fr][8 * bc[v] + 2 * fk + h] = xj[v][h];
                        }
                    __syncthreads();
                };
                __syncthreads();
                // the solved panel blocks: X = A M, and to refine them R = A - X L^T, X + R M
                multiply(s_pi, s_pj, s_m, 1.0);
                if (refine) {
                    for (int e = tid; e < kCB * kCB; e += kCThreads) s_l[e / kCB][e % kCB] = __ldcg(q.Li + (size_t)kb * kCB * kCB + e);
                    keep(s_xi, s_xj);
                    fetch(s_pi, s_pj);
                    multiply(s_xi, s_xj, s_l, -1.0);
                    keep(s_pi, s_pj);
                    fetch(s_xi, s_xj);
                    multiply(s_pi, s_pj, s_m, 1.0);
                }
                __syncthreads();
                keep(s_pi, s_pj);
                double h0[2][2] = {};
                const double (*sj)[kCPitch] = two ? s_pj : s_pi;
#pragma unroll
                for (int k = 0; k < kCB; k += 4) {
                    const double x = -s_pi[8 * br + fr][k + fk];
#pragma unroll
                    for (int v = 0; v < 2; ++v) dmma(k & 4 ? h0[v] : g[v], x, sj[8 * bc[v] + fr][k + fk]);
                }
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    g[v][0] += h0[v][0];
                    g[v][1] += h0[v][1];
                    *reinterpret_cast<double2*>(G + (size_t)(i0 + 8 * br + fr) * Np + j0 + 8 * bc[v] + 2 * fk) = make_double2(g[v][0], g[v][1]);
                }
                if (jb == kb + 1) {
                    for (int e = tid; e < kCB * kCB; e += kCThreads) G[(size_t)(k0 + e / kCB) * Np + i0 + e % kCB] = s_pi[e % kCB][e / kCB];
                    if (i0 <= N && N < i0 + kCB && tid < kCB) q.z[k0 + tid] = s_pi[N - i0][tid];
                }
                __syncthreads();
                if (b == 0) {                                // the next diagonal block, whole
#pragma unroll
                    for (int v = 0; v < 2; ++v)
#pragma unroll
                        for (int h = 0; h < 2; ++h) s_pi[8 * br + fr][8 * bc[v] + 2 * fk + h] = g[v][h];
                    __syncthreads();
                }
            }
            if (b == 0) factor(kb + 1);                      // before the barrier
        }
        grid.sync();
    }
    if (blockIdx.x != 0) return;

    // L^T a = z, from the last block up: a_kb = M_kb (z_kb - sum of L_i,kb^T a_i over the blocks i below).  Row k0 + j of the upper
    // triangle holds L's column.  The first warp finishes a block from what the others brought in and summed a phase earlier: the factor and its
    // inverse, the block of L next to the diagonal, and the part of the sums whose a_i were known then.
    if (warp == 0 && lane == 0 && !good) *q.status = 1;
    __shared__ double s_sum[2][kCB];
    __shared__ bool s_refine[2];
    double (*s_inv)[kCPitch] = s_m, (*s_next)[kCPitch] = s_m + 2 * kCB, (*s_own)[kCPitch] = s_m + 4 * kCB;   // two of each
    double* s_a = reinterpret_cast<double*>(s_m + 6 * kCB);
    const int nblk = (N + kCB - 1) / kCB;
    constexpr int kHelpers = kCThreads / 32 - 1;
    auto bring = [&](int kb) {                               // for block kb, by warps 1 .. 7, while a of blocks above kb + 1 is known
        const int k0 = kb * kCB, buf = kb & 1, w = warp - 1;
        constexpr int kEach = (kCB * kCB + kCThreads - 33) / (kCThreads - 32);
        const bool refine = __ldcg(q.refine + kb) != 0;
        double inv[kEach], next[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            const int e = min(tid - 32 + u * (kCThreads - 32), kCB * kCB - 1), r = e / kCB, c = e % kCB;
            inv[u] = __ldcg(q.Mi + (size_t)kb * kCB * kCB + e);
            next[u] = __ldcg(G + (size_t)(k0 + r) * Np + min(k0 + kCB + c, Np - 1));   // past column N: not used
        }
        // five rows a warp, side by side: what counts is how many loads are on their way
        constexpr int kRows = (kCB + kHelpers - 1) / kHelpers;
        double sum[kRows];
        const double* row[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            sum[u] = 0.0;
            row[u] = G + (size_t)min(k0 + w + kHelpers * u, N - 1) * Np;   // rows past the last are not used
        }
#pragma unroll 4
        for (int i = k0 + 2 * kCB + lane; i < N; i += 32) {
            const double ai = s_a[i];
#pragma unroll
            for (int u = 0; u < kRows; ++u) sum[u] += __ldcg(row[u] + i) * ai;
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], o);
            if (lane == 0 && w + kHelpers * u < kCB) s_sum[buf][w + kHelpers * u] = sum[u];
        }
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            const int e = min(tid - 32 + u * (kCThreads - 32), kCB * kCB - 1), r = e / kCB, c = e % kCB;
            s_inv[buf * kCB + r][c] = inv[u];
            if (refine) s_own[buf * kCB + r][c] = __ldcg(q.Li + (size_t)kb * kCB * kCB + e);
            s_next[buf * kCB + r][c] = next[u];
        }
        if (tid == 32) s_refine[buf] = refine;
    };
    __syncthreads();
    if (warp > 0) bring(nblk - 1);
    __syncthreads();
    for (int kb = nblk - 1; kb >= 0; --kb) {
        const int k0 = kb * kCB, ncols = min(kCB, N - k0), buf = kb & 1;
        if (warp == 0) {
            double v = 0.0;
            if (lane < ncols) {
                v = __ldcg(q.z + k0 + lane) - s_sum[buf][lane];
                const int below = min(kCB, N - k0 - kCB);
                double u[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
                for (int c = 0; c < below; ++c) u[c & 3] += s_next[buf * kCB + lane][c] * s_a[k0 + kCB + c];
                v -= (u[0] + u[1]) + (u[2] + u[3]);
            }
            // row `lane` of a block of the buffer times a vector in s_t
            auto times = [&](const double (*m)[kCPitch], int at, double x) {
                __syncwarp();
                s_t[at][lane] = x;
                __syncwarp();
                double u[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int c = 0; c < kCB; ++c) u[c & 3] += m[buf * kCB + lane][c] * s_t[at][c];
                return lane < ncols ? (u[0] + u[1]) + (u[2] + u[3]) : 0.0;
            };
            double a = times(s_inv, 0, v);
            if (s_refine[buf]) a += times(s_inv, 2, v - times(s_own, 1, a));
            if (lane < ncols) {
                s_a[k0 + lane] = a;
                q.a[k0 + lane] = a;
            }
        } else if (kb > 0) {
            bring(kb - 1);
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
constexpr size_t kKeepBytes = (size_t)144 << 20;
constexpr size_t kLeastDigitBytes = (size_t)32 << 20;   // digits are not divided further for that
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
    const size_t chol_smem = (size_t)(kCSmem + N) * sizeof(double);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ridge_cholesky_solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)((kCSmem + ROCKET_RIDGE_MAX_EXAMPLES) * sizeof(double)));
    if (e != cudaSuccess) return status_of(e);
    const int col_blocks = (P + 31) / 32;
    const int nt = (N + kGT - 1) / kGT, tiles = nt * (nt + 1) / 2;
    const int nb = (N + 1 + kCB - 1) / kCB, Np = nb * kCB;
    // Integers on the tensor cores beyond N N P = 3e8 (us, FP64 and integers: 200 x 4,000 143 and 148, 300 x 3,000 171 and 175, 677 x 300 293 and 298;
    // 677 x 800 306 and 308; 200 x 8,000 168 and 154, 100 x 40,000 217 and 209, 300 x 5,000 193 and 186, 677 x 20,000 784 and 546).  Their tiles are 128
    // rows high: up to 64 rows are half empty, and the digits of as many columns take longer than the products (64 x 120,000 364 and 398,
    // 24 x 300,000 474 and 878).
    bool integers = N > 64 && (double)N * N * P >= 3e8;
    GramPlan gram{};
    int slices = 0, slice = 0;
    size_t o_mu, o_a, o_part, o_ybar, o_G, o_Mi, o_Li, o_refine, o_z, o_gram, o_int, o_up, o_down, o_digits, bytes;
    // workspace: mu[P], a[N], part[col_blocks], ybar, G[Np][Np], Mi[nb][32][32], Li[nb][32][32], refine[nb], z[Np], partial Gram tiles, ticket, status; for
    // integers the rows' scales and digits
    auto lay_out = [&]() {
        size_t off = 0;
        auto take = [&](size_t doubles) { const size_t o = off; off += (doubles + 31) / 32 * 32; return o; };
        o_mu = take(P); o_a = take(N); o_part = take(col_blocks); o_ybar = take(1); o_G = take((size_t)Np * Np);
        o_Mi = take((size_t)nb * kCB * kCB); o_Li = take((size_t)nb * kCB * kCB); o_refine = take((nb + 1) / 2); o_z = take(Np); o_gram = take((size_t)slices * tiles * kGT * kGT); o_int = take(2);
        o_up = take(integers ? N : 0); o_down = take(integers ? N : 0); o_digits = take(integers ? gram.digit_bytes / sizeof(double) : 0);
        bytes = off * sizeof(double);
    };
    FitWorkspace ws;
    if (integers) {
        auto plan = [&](size_t digits) {
            gram = gram_plan(N, P, sms, digits);
            slices = gram.slices;
            lay_out();
        };
        plan(kGramDigitBytes);
        // Digits of fewer columns at a time where that lets the workspace be the one that is kept: two or three chunks cost little, allocations a
        // millisecond (1,600 x 20,000).
        const bool could = bytes <= kKeepBytes + gram.digit_bytes - std::min(gram.digit_bytes, kLeastDigitBytes);
        while (could && bytes > kKeepBytes && gram.digit_bytes > kLeastDigitBytes) plan(gram.digit_bytes / 4 * 3);
        if ((e = ws.take(bytes)) == cudaErrorMemoryAllocation) {   // no room for the digits: the FP64 kernel, which needs none
            cudaGetLastError();
            integers = false;
        }
    }
    if (!integers) {
        // Slices of the feature axis: about two waves of the four blocks an SM holds, at least 128 columns each, and no more
        // than 40 MB of partial tiles (or one slice, 65 MB at the most examples).
        const size_t tile_bytes = (size_t)kGT * kGT * sizeof(double);
        slices = std::max(1, std::min({8 * sms / tiles, P / 128, (int)(((size_t)40 << 20) / (tile_bytes * tiles))}));
        slice = ((P + slices - 1) / slices + kGP - 1) / kGP * kGP;
        slices = (P + slice - 1) / slice;
        lay_out();
        e = ws.take(bytes);
    }
    if (e != cudaSuccess) return status_of(e);
    double* d = static_cast<double*>(ws.ptr);
    unsigned* ticket = reinterpret_cast<unsigned*>(d + o_int);
    int* status = reinterpret_cast<int*>(d + o_int + 1);
    ridge_means_kernel<<<col_blocks + 1, kRThreads, 0, stream>>>(feat_dev, y_dev, N, P, d + o_mu, d + o_ybar, ticket, status + 1);
    if (integers)
        e = launch_gram(gram, feat_dev, N, P, d + o_mu, d + o_up, d + o_down, reinterpret_cast<uint8_t*>(d + o_digits), d + o_gram, status + 1, stream);
    else
        ridge_gram_kernel<<<dim3(tiles, slices), kGThreads, gram_smem, stream>>>(feat_dev, N, P, d + o_mu, slice, d + o_gram);
    CholArgs q{d + o_gram, slices, tiles, (double)alpha, y_dev, d + o_ybar, d + o_G, d + o_Mi, d + o_Li, reinterpret_cast<int*>(d + o_refine), d + o_z, d + o_a, status, N, Np};
    void* args[] = {&q};
    // one block per SM: more would lengthen the grid barriers without shortening the chain
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(ridge_cholesky_solve_kernel),
                                    dim3((unsigned)std::max(1, std::min(sms, nb * (nb + 1) / 2))), dim3(kCThreads), args, chol_smem, stream);
    ridge_weights_kernel<<<col_blocks, kRThreads, 0, stream>>>(feat_dev, N, P, d + o_mu, d + o_a, d + o_ybar, w_dev, b_dev,
                                                               d + o_part, ticket);
    count_launch(integers ? 3 : 4);                        // launch_gram counts its own
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
