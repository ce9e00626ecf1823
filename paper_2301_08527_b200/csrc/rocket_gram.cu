// Gram matrix of the centred features on the fifth-generation tensor cores, in integers.
//
// Fc = F - mu is taken in double precision, every row scaled by a power of two so that its largest magnitude lies in [63/64 2^54, 63/64 2^55),
// rounded to an integer and written as seven signed base-256 digits, d_0 first.  Then G_ij is a sum of digit products: all with a + b <= 7 are kept
// (34 of 49), products with the same a + b share a 32-bit accumulator and are exact there (7 * 16,384 columns * 128^2 < 2^31), and the eight
// accumulators meet in double precision.
//
// How close: what is left out and the rounding to integers together are of the order of 2^-54 |x_i| |x_j| for rows x_i, x_j of Fc, below the 2^-53 that
// the factorisation rounds its own terms by.  With a + b <= 6 (28 products) 2^-47 max|x_i| max|x_j| was left out: no matter among values of one
// size, but the weights of 120 examples of 10,000 shares and maxima, one column of them 10^6 times as large, were off by 1.0e-5 where sums in FP64
// leave 1.2e-6; they are off by 3.0e-7 now.
//
// Why: FP64 products run at 37 TFLOP/s at the most, 8-bit ones at a hundred times that, and 34 of those replace one.  Measured at 677 x
// 20,000: 254 us (scales 21, digits 28, products 205; 28 products took 180) where FP64 matrix instructions took 496.
#include <cstdint>

#include "rocket_fast_dev.cuh"
#include "rocket_gram.h"
#include "rocket_internal.h"

namespace rocket {
namespace {

using fast::bulk_g2s;
using fast::mbar_arrive_expect_tx;
using fast::mbar_init;
using fast::mbar_wait;
using fast::smem_u32;

constexpr int kDigits = kGramDigits, kSums = 8, kTileM = kGramTileM, kTileN = kGramTileN, kStageK = kGramStageK;
// The digits lie in memory as the matrix instruction reads them from shared memory (8 rows x 16 bytes to a core matrix, no swizzle):
// [block of 64 columns][group of 8 rows][digit][4 core matrices][8 rows][16 columns], so that the operands of a stage are two bulk copies.
constexpr int kCoreBytes = 128, kDigitBytes = kStageK / 16 * kCoreBytes, kGroupBytes = kGramGroupBytes;
static_assert(kGroupBytes == kDigits * kDigitBytes, "a group's digits");
constexpr int kABytes = kTileM / 8 * kGroupBytes, kBBytes = kTileN / 8 * kGroupBytes, kStageBytes = kABytes + kBBytes;
constexpr int kStages = 2, kGramThreads = 128;
static_assert(kSums * kTileN <= 512, "an accumulator per a + b");

// up[i] = 2^k with up[i] max_p |F[i][p] - mu[p]| in [63/64 2^54, 63/64 2^55), as large as seven signed digits hold; down[i] = 1 / up[i]; NaN where
// a value of the row is not finite.
__global__ void __launch_bounds__(256)
gram_scale_kernel(const float* __restrict__ F, int P, const double* __restrict__ mu, double* __restrict__ up, double* __restrict__ down) {
    __shared__ unsigned long long s_max;
    if (threadIdx.x == 0) s_max = 0ull;
    __syncthreads();
    const float* __restrict__ f = F + (size_t)blockIdx.x * P;
    unsigned long long m = 0ull;                       // magnitudes compare as integers, infinities and NaN above all others
#pragma unroll 8
    for (int p = threadIdx.x; p < P; p += 256)
        m = max(m, (unsigned long long)__double_as_longlong((double)__ldg(f + p) - __ldg(mu + p)) & 0x7fffffffffffffffull);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, m);
    __syncthreads();
    if (threadIdx.x > 0) return;
    m = s_max;
    const int e = (int)(m >> 52) - 1022 + ((m >> 46 & 63ull) == 63ull ? 1 : 0);   // the maximum is below 63/64 2^e
    const int k = min(max(55 - e, -1022), 1022);
    const bool finite = (m >> 52) < 2047ull;
    up[blockIdx.x] = finite ? __longlong_as_double((long long)(1023 + k) << 52) : __longlong_as_double(0x7ff8000000000000ll);
    down[blockIdx.x] = finite ? __longlong_as_double((long long)(1023 - k) << 52) : __longlong_as_double(0x7ff8000000000000ll);
}

// The digits of columns [p0, p0 + 64 blocks): a warp writes a core matrix of every digit, 128 contiguous bytes each.  Zeros past the last
// row and column.
__global__ void __launch_bounds__(256)
gram_digits_kernel(const float* __restrict__ F, int N, int P, int p0, int cores, const double* __restrict__ mu, const double* __restrict__ up, int groups,
                   uint8_t* __restrict__ digits) {
    const int lane = threadIdx.x & 31, core = blockIdx.x * 8 + (threadIdx.x >> 5), group = blockIdx.y;
    const int row = group * 8 + lane / 4, k = core * 16 + lane % 4 * 4;
    if (core >= cores) return;
    unsigned lo[4], hi[4];
    const bool there = row < N;
    const double scale = there ? __ldg(up + row) : 0.0;
    const float* __restrict__ f = F + (size_t)(there ? row : 0) * P + p0 + k;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const bool ok = there && p0 + k + c < P;
        const double x = ok ? (double)__ldg(f + c) - __ldg(mu + p0 + k + c) : 0.0;
        // with 128 added to every digit the digits are the bytes
        const unsigned long long q = (unsigned long long)__double2ll_rn(x * scale) + 0x80808080808080ull;
        lo[c] = (unsigned)q;
        hi[c] = (unsigned)(q >> 32);
    }
    uint8_t* out = digits + ((size_t)(core >> 2) * groups + group) * kGroupBytes + (core & 3) * kCoreBytes + 4 * lane;
#pragma unroll
    for (int a = 0; a < kDigits; ++a) {
        const int byte = kDigits - 1 - a;
        const unsigned* w = byte < 4 ? lo : hi;
        const unsigned sel = (byte & 3) | ((byte & 3) + 4) << 4;
        const unsigned v = __byte_perm(__byte_perm(w[0], w[1], sel), __byte_perm(w[2], w[3], sel), 0x5410);
        *reinterpret_cast<unsigned*>(out + a * kDigitBytes) = v ^ 0x80808080u;
    }
}

struct GramArgs {
    const uint8_t* digits;
    const double* down;
    double* part;             // [slices][tiles of 64 x 64][64][64]
    int* failed;
    int N, groups, blocks, tiles, slices, add;   // groups: of 8 rows; blocks: of 64 columns, no fewer than slices; tiles: 64 x 64 ones of a slice; add: onto what part holds
};

__device__ __forceinline__ uint64_t operand(uint32_t at) {   // K-major, no swizzle: core matrices along K, groups of 8 rows
    return (uint64_t)((at & 0x3ffffu) >> 4) | (uint64_t)(kCoreBytes >> 4) << 16 | (uint64_t)(kGroupBytes >> 4) << 32 | 1ull << 46;
}

// One 128 x 64 tile of the lower triangle over a slice of the columns.  One thread copies stages in, one issues the matrix instructions
// (68 per stage of 64 columns), all four warps turn the accumulators into doubles.  Bound: the matrix pipe, an instruction of 128 x 64 x 32
// every 70 clocks; with A's digits copied to tensor memory, which spares two thirds of the shared-memory reads, the same.
__global__ void __launch_bounds__(kGramThreads, 1)
gram_mma_kernel(const GramArgs a) {
    extern __shared__ __align__(128) unsigned char gram_smem[];
    __shared__ __align__(8) unsigned long long s_full[kStages], s_empty[kStages], s_done;
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t full0 = smem_u32(s_full), empty0 = smem_u32(s_empty), done = smem_u32(&s_done);
    const uint32_t raw = smem_u32(gram_smem), stage0 = (raw + 127u) & ~127u;
    int bi = (int)((sqrtf(4.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
    while (bi * (bi + 1) > (int)blockIdx.x) --bi;
    while ((bi + 1) * (bi + 2) <= (int)blockIdx.x) ++bi;
    const int bj = (int)blockIdx.x - bi * (bi + 1);
    const int kb0 = (int)((long long)a.blocks * blockIdx.y / a.slices), n_st = (int)((long long)a.blocks * (blockIdx.y + 1) / a.slices) - kb0;
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8u * i, 1);
            mbar_init(empty0 + 8u * i, 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    bool ok = true;

    if (tid == 0) {                                    // copies
        int st = 0;
        for (; st < n_st; ++st) {
            const int slot = st % kStages;
            if (st >= kStages && !(ok = mbar_wait(empty0 + 8u * slot, (st / kStages - 1) & 1))) break;
            const uint8_t* src = a.digits + (size_t)(kb0 + st) * a.groups * kGroupBytes;
            const uint32_t dst = stage0 + slot * kStageBytes, bar = full0 + 8u * slot;
            mbar_arrive_expect_tx(bar, kStageBytes);
            bulk_g2s(dst, src + (size_t)bi * kABytes, kABytes, bar);
            bulk_g2s(dst + kABytes, src + (size_t)bj * kBBytes, kBBytes, bar);
        }
        if (!ok)                                       // what was started has to land before the block ends
            for (int i = max(0, st - kStages); i < st; ++i) mbar_wait(full0 + 8u * (i % kStages), (i / kStages) & 1);
    } else if (tid == 32) {                            // multiplications
        // D: 32-bit integers; A, B: signed bytes, K-major; 128 x 64
        constexpr uint32_t kInstr = 2u << 4 | 1u << 7 | 1u << 10 | (uint32_t)(kTileN >> 3) << 17 | (uint32_t)(kTileM >> 4) << 24;
        for (int st = 0; st < n_st; ++st) {
            const int slot = st % kStages;
            if (!(ok = mbar_wait(full0 + 8u * slot, (st / kStages) & 1))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t at = stage0 + slot * kStageBytes;
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int da = 0; da < kDigits; ++da)
#pragma unroll
                    for (int db = 0; db < kDigits && db + da < kSums; ++db) {
                        // the first product of an accumulator assigns it
                        const uint32_t fresh = (da == 0 || db == kDigits - 1) && k == 0 && st == 0 ? 0u : 1u;
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                            ::"r"(tmem + (uint32_t)((da + db) * kTileN)), "l"(operand(at + da * kDigitBytes + k * 2 * kCoreBytes)),
                            "l"(operand(at + kABytes + db * kDigitBytes + k * 2 * kCoreBytes)), "r"(kInstr), "r"(fresh) : "memory");
                    }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty0 + 8u * slot) : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done) : "memory");
    }
    __syncwarp();
    ok = mbar_wait(done, 0) && ok;
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok && tid == 0) atomicExch(a.failed, 1);

    // warp w holds rows 32 w .. 32 w + 31 of the tile, a row per lane
    const int i = bi * kTileM + tid, ti = i / 64, j0 = bj * kTileN;
    const double di = i < a.N ? __ldg(a.down + i) : 0.0;
    double* out = a.part + ((size_t)blockIdx.y * a.tiles + (size_t)ti * (ti + 1) / 2 + bj) * 4096 + (i % 64) * 64;
    const bool lower = bj <= ti && i < (a.N + 63) / 64 * 64;
#pragma unroll 1
    for (int c = 0; c < kTileN; c += 8) {
        uint32_t v[kSums][8];
#pragma unroll
        for (int s = 0; s < kSums; ++s)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(v[s][0]), "=r"(v[s][1]), "=r"(v[s][2]), "=r"(v[s][3]), "=r"(v[s][4]), "=r"(v[s][5]), "=r"(v[s][6]), "=r"(v[s][7])
                         : "r"(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(s * kTileN + c)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (!lower) continue;
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            double g[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                double sum = 0.0;                      // smallest first
#pragma unroll
                for (int s = kSums - 1; s >= 0; --s) sum = fma(sum, 1.0 / 256.0, (double)(int)v[s][e + h]);
                const int j = j0 + c + e + h;
                // 256^6 per factor between the leading digit and the integer
                g[h] = sum * (281474976710656.0 * di) * (281474976710656.0 * (j < a.N ? __ldg(a.down + j) : 0.0));
            }
            double2* to = reinterpret_cast<double2*>(out + c + e);
            if (a.add) {
                const double2 old = *to;
                *to = make_double2(old.x + g[0], old.y + g[1]);
            } else {
                *to = make_double2(g[0], g[1]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

constexpr size_t kGramSmem = (size_t)kStages * kStageBytes + 128;

}  // namespace

cudaError_t launch_gram(const GramPlan& g, const float* F, int N, int P, const double* mu, double* up, double* down, uint8_t* digits, double* part,
                        int* failed, cudaStream_t stream) {
    cudaError_t e = cudaFuncSetAttribute(gram_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGramSmem);
    if (e != cudaSuccess) return e;
    gram_scale_kernel<<<N, 256, 0, stream>>>(F, P, mu, up, down);
    count_launch();
    const int nt = (N + 63) / 64, blocks = (P + kStageK - 1) / kStageK;
    for (int b0 = 0; b0 < blocks; b0 += g.chunk) {
        const int nb = std::min(g.chunk, blocks - b0);
        gram_digits_kernel<<<dim3((nb * 4 + 7) / 8, g.groups), 256, 0, stream>>>(F, N, P, b0 * kStageK, nb * 4, mu, up, g.groups, digits);
        const int slices = gram_slices(g, nb);
        const GramArgs a{digits, down, part, failed, N, g.groups, nb, nt * (nt + 1) / 2, slices, b0 > 0 ? 1 : 0};
        gram_mma_kernel<<<dim3(g.blocks_mn, slices), kGramThreads, kGramSmem, stream>>>(a);
        count_launch(2);
    }
    return cudaGetLastError();
}

}  // namespace rocket
