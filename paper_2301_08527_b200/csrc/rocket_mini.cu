// MINIROCKET on the device (the extension the paper names in Section 6: "the PyTorch GPU implementation could
// be extended to the MINIROCKET model"; Section 2 describes the model: two-valued kernels from a fixed set,
// biases sampled from the input data, PPV as the only pooled feature).
//
//   parameters   built on the host from one seed (rocket_mini_create): 84 kernels of length 9 with three taps
//                of weight 2 and six of weight -1, dilations floor(2^x) spread up to (L - 1) / 8, padding 4 d on
//                every other (dilation, kernel) combination, a random channel subset per combination
//   fit          rocket_mini_fit, on the host (a one-off over one training example per combination): the bias of
//                a feature is a quantile of the combination's convolution output on that example
//   transform    rocket_mini_transform, one fused kernel of two (the other: rocket_mini_walk.cuh): a block stages a tile of the dilated view with all the
//                channels that the combinations of a dilation use, its warps take the combinations one by one -
//                channels summed, nine-tap convolution, comparison with every bias of the combination, all in
//                registers - so the convolution outputs never reach memory; a small kernel then turns counts into
//                shares of outputs (Eq. 1-2 against the bias)
//
// The kernel weights take two values, so every product is one fused multiply-add with -1 or 2: on this
// hardware an addition and a fused multiply-add take the same issue slot, and the additions-only form that
// speeds the method up on a CPU brings nothing here.
#include <algorithm>
#include <array>
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <numeric>
#include <thread>
#include <vector>

#include "rocket_fast.h"
#include "rocket_fast_dev.cuh"
#include "rocket_fast_geom.h"
#include "rocket_internal.h"
#include "rocket_mini_walk.cuh"

namespace rocket {
namespace fast {
namespace {

constexpr int kKernels = 84, kLen = 9;
constexpr int kMRows = 14, kMInRows = kMRows + kLen - 1;      // output rows of a tile, input rows
constexpr int kMWarps = 20, kMThreads = 32 * kMWarps;
constexpr int kMProducers = 3;                                // producer warps of the double-buffered form
constexpr int kMPlanes = 20, kMPlanesWide = 2 * kMPlanes;     // (example, channel) planes of a tile: two tiles in shared memory, or one
constexpr int kMPlaneFloats = kMInRows * kWarpCols, kMPlaneBytes = kMPlaneFloats * 4;
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kStreamBase = 1ull << 32;
constexpr double kInvGoldenRatio = 0.6180339887498949;

inline uint64_t mix(uint64_t z) {   // splitmix64 finaliser
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
inline uint64_t draw_u64(uint64_t seed, uint64_t stream, uint64_t slot) {
    return mix(mix(seed + kGolden * (stream + 1)) + kGolden * (slot + 1));
}
inline double draw_uniform(uint64_t seed, uint64_t stream, uint64_t slot) {
    return static_cast<double>(draw_u64(seed, stream, slot) >> 11) * 0x1.0p-53;
}

// One combination (32 words): its outputs are u = t d + r with tl d <= u < th d + rh (A[t][r] = x[t d + r]).
struct alignas(16) MiniRec {
    int32_t m, f0, nf, tl, th, rh, pad_[2];
    int32_t ch[kLen];                     // byte offsets of the channels' planes in a tile
    float w[kLen];                        // the weights, negated
    int32_t pad2_[6];
};
static_assert(sizeof(MiniRec) == 128, "MiniRec must be 32 words");
// Combinations [kbeg, kend) of one dilation that use at most kMPlanes channels between them, kMPlanesWide in a handle whose
// tiles have shared memory to themselves (64 words).
struct alignas(16) MiniBucket {
    int32_t d, raster_len, kbeg, kend, nch, pad_[7];
    int32_t ch[kMPlanesWide], pad2_[12];
};
static_assert(sizeof(MiniBucket) == 256, "MiniBucket must be 64 words");
// 64 consecutive columns of a bucket's raster: bands of kMRows rows of A, strung together band by band.
struct MiniTile { int32_t bucket, c0; };

struct MiniArgs {
    const float* X;
    const MiniRec* recs;
    const MiniBucket* buckets;
    const MiniTile* tiles;
    const float* bias;
    int* counts;                          // [N][F]: the features while they are counts
    int* failed;                          // the call's flag
    int N, C, L, F, n_tiles;
    int examples, groups, parts;          // examples of a tile, groups of examples, parts a tile's combinations are dealt in
};

// A tile as the producers describe it to the consumers.
struct TileAt { int d, raster_len, plane_bytes, c0, n0, ne, kbeg, n_work; };   // plane_bytes: of one example's planes

// *p, or zero; the loads stay in the order they are written in.
__device__ __forceinline__ float load_if(const float* p, unsigned ok) {
    float v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@q ld.global.nc.f32 %0, [%1];\n\t}" : "=f"(v) : "l"(p), "r"(ok));
    return v;
}

// The columns lane and lane + 32 of a tile: their first position (64 bits: columns that do not exist lie anywhere), and the input
// rows that lie in the series.
struct FillAt {
    int d;
    long long u0, u1;
    unsigned in0, in1;
    bool inside;
    __device__ __forceinline__ FillAt(int d_, int raster_len, int c0, int L, int lane) : d(d_) {
        const int cg0 = c0 + lane, cg1 = cg0 + 32, band0 = (int)((unsigned)cg0 / (unsigned)d), band1 = (int)((unsigned)cg1 / (unsigned)d);
        const int t0 = band0 * kMRows - 4, t1 = band1 * kMRows - 4, r0 = cg0 - band0 * d, r1 = cg1 - band1 * d;
        const int th = (int)((unsigned)L / (unsigned)d), rh = L - th * d;
        u0 = (long long)t0 * d + r0;
        u1 = (long long)t1 * d + r1;
        int lo, hi;
        rows_in_series(t0, r0, th, rh, kMInRows, lo, hi);
        in0 = cg0 < raster_len ? row_mask(lo, hi) : 0u;
        rows_in_series(t1, r1, th, rh, kMInRows, lo, hi);
        in1 = cg1 < raster_len ? row_mask(lo, hi) : 0u;
        constexpr unsigned kAll = (1u << kMInRows) - 1u;
        inside = __all_sync(kFull, (in0 & in1) == kAll);
    }
};

// Planes warp, warp + warps, .. of a tile: the bucket's nch channels of ne examples, zeros outside the series.  All of a plane's
// loads come before its stores: of 4-byte asynchronous copies a warp keeps only a few in flight, and with them four warps took
// 35 thousand clocks for a tile.
template <class Channel>
__device__ __forceinline__ void fill_planes(const MiniArgs& a, const FillAt& at, float* to, Channel channel, int nch, int n0, int ne,
                                            int warp, int warps, int lane) {
    for (int pl = warp; pl < nch * ne; pl += warps) {
        const int e = pl / nch, c = pl - e * nch;
        const float* __restrict__ src = a.X + ((size_t)(n0 + e) * a.C + channel(c)) * a.L;
        float* dst = to + pl * kMPlaneFloats + lane;
        float v0[kMInRows], v1[kMInRows];
        const float* __restrict__ p0 = src + at.u0;
        const float* __restrict__ p1 = src + at.u1;
        if (at.inside) {
#pragma unroll
            for (int s = 0; s < kMInRows; ++s) {
                v0[s] = __ldg(p0);
                v1[s] = __ldg(p1);
                p0 += at.d;
                p1 += at.d;
            }
        } else {
#pragma unroll
            for (int s = 0; s < kMInRows; ++s) {
                v0[s] = load_if(p0, at.in0 >> s & 1);
                v1[s] = load_if(p1, at.in1 >> s & 1);
                p0 += at.d;
                p1 += at.d;
            }
        }
#pragma unroll
        for (int s = 0; s < kMInRows; ++s) {
            dst[s * kWarpCols] = v0[s];
            dst[s * kWarpCols + 32] = v1[s];
        }
    }
}

// How many of the 2 x 14 outputs exceed a bias: the signs of bias - z (exact: the difference of two floats rounds to zero only
// when they are equal).  acc = -z.
__device__ __forceinline__ int mini_count(const u64 (&acc)[kMRows], float b) {
    const u64 bp = pack2(b, b);
    unsigned s0 = 0, s1 = 0;              // two chains
#pragma unroll
    for (int o = 0; o < kMRows; ++o) {
        float x, y;
        unpack2(add2(acc[o], bp), x, y);
        s0 = __funnelshift_l(__float_as_uint(x), s0, 1);
        s1 = __funnelshift_l(__float_as_uint(y), s1, 1);
    }
    return __popc(s0 | s1 << kMRows);
}

// Bound: shared memory (67 % of its wavefronts at 60 x 20 x 50,000) and instruction issue (59 %) together - per pair of outputs 9 packed multiply-adds, (m - 1) 22/14 packed adds and m 22/14 loads for the
// channel sums (m channels, 3.9 on average) and, per bias (3.8 on average), a packed add and two shifts that collect the signs
// of bias - z.  What the layout is for: the channels of a tile are read once for the 84 combinations of a dilation (one
// combination per block and tile, the earlier form, read 146 GB from L2 for 60 x 20 x 50,000), the packed operations work on
// two columns at a time, and two tiles are in shared memory: producer warps bring the next one in while the others work on this
// one, and a warp that finds no combination left goes on to the next tile without waiting.  Measured (the earlier form 17.3 ms):
// 10.4 ms for 60 x 20 x 50,000 and 9,996 features (12 rows: 10.75, of which 9.9 remain without the copies into shared memory;
// the shared memory's bandwidth counts, so the tile is as high as two of them fit: 22 input rows for 14 rows of outputs).
template <bool WIDE>
__global__ void __launch_bounds__(kMThreads, 1) mini_tile_kernel(const __grid_constant__ MiniArgs a) {
    constexpr int kConsumers = WIDE ? kMWarps : kMWarps - kMProducers;
    extern __shared__ __align__(128) float planes[];              // [2][kMPlanes][kMInRows][64]
    __shared__ unsigned long long s_full[2], s_empty[2];
    __shared__ TileAt s_tile[2];
    __shared__ int s_pos;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(kFull, tid >> 5, 0);
    const uint32_t full0 = smem_u32(s_full), empty0 = smem_u32(s_empty);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(full0 + 8u * i, 32 * kMProducers + 1);
            mbar_init(empty0 + 8u * i, kConsumers);
        }
        s_pos = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // The block's tiles: items blockIdx.x, blockIdx.x + gridDim.x, .. of all (tile, part, group of examples).  The (combination,
    // example) pairs of the block's tiles form one sequence that the consumer warps draw from.
    const unsigned total = (unsigned)a.groups * (unsigned)a.n_tiles * (unsigned)a.parts;
    const int K = (int)((total - blockIdx.x + gridDim.x - 1) / gridDim.x);
    auto word = [](int v, int i) { return __shfl_sync(kFull, v, i); };
    bool ok = true;

    if (!WIDE && warp >= kConsumers) {
        // ---- producers: every channel of the bucket, a plane per warp, zeros outside the series
        const unsigned per_group = (unsigned)a.n_tiles * (unsigned)a.parts;
        auto tile_of = [&](int k) { return (blockIdx.x + (unsigned)k * gridDim.x) % per_group / (unsigned)a.parts; };
        int2 at = __ldg(reinterpret_cast<const int2*>(a.tiles + tile_of(0)));
        int words = __ldg(reinterpret_cast<const int*>(a.buckets + at.x) + lane);
        for (int k = 0; k < K; ++k) {
            const unsigned g = blockIdx.x + (unsigned)k * gridDim.x, group = g / per_group;
            const int part = (int)(g % per_group % (unsigned)a.parts);
            const int d = word(words, 0), raster_len = word(words, 1), nch = word(words, 4), c0 = at.y, bucket_words = words;
            const int n0 = (int)group * a.examples, ne = min(a.examples, a.N - n0), first = word(words, 2);
            const int combos = word(words, 3) - first, beg = combos * part / a.parts, end = combos * (part + 1) / a.parts;
            if (k + 1 < K) at = __ldg(reinterpret_cast<const int2*>(a.tiles + tile_of(k + 1)));     // on its way
            const FillAt at_columns(d, raster_len, c0, a.L, lane);
            if (k >= 2 && !(ok = mbar_wait(empty0 + 8u * (k & 1), ((k - 2) >> 1) & 1))) break;
            if (tid == 32 * kConsumers) {
                s_tile[k & 1] = TileAt{d, raster_len, nch * kMPlaneBytes, c0, n0, ne, first + beg, (end - beg) * ne};
                mbar_arrive(full0 + 8u * (k & 1));
            }
            if (k + 1 < K) words = __ldg(reinterpret_cast<const int*>(a.buckets + at.x) + lane);
            fill_planes(a, at_columns, planes + (k & 1) * kMPlanes * kMPlaneFloats, [&](int c) { return word(bucket_words, 12 + c); }, nch, n0, ne, warp - kConsumers, kMProducers, lane);
            mbar_arrive(full0 + 8u * (k & 1));
        }
        if (!ok && lane == 0) atomicExch(a.failed, 1);
        return;
    }

    // ---- consumers
    auto draw = [&]() {
        int p = 0;
        if (lane == 0) p = atomicAdd(&s_pos, 1);
        return __shfl_sync(kFull, p, 0);
    };
    auto load_rec = [&](const TileAt& t, int w) {
        return __ldg(reinterpret_cast<const int*>(a.recs + t.kbeg + (t.ne == 1 ? w : w / t.ne)) + lane);
    };
    TileAt cur{};
    int k = 0, base = 0;
    int pos = draw();
    // the lane's two columns of the tile: band of rows and column of A
    int trow0 = 0, trow1 = 0, c0 = 0, c1 = 0;
    bool ok0 = false, ok1 = false;
    int rec_next = 0;                                  // the record of the pair at pos, on its way
    auto fetch_rec = [&]() {
        if (pos < base + cur.n_work) rec_next = load_rec(cur, pos - base);
    };
    auto enter = [&]() {
        if constexpr (WIDE) {
            const unsigned g = blockIdx.x + (unsigned)k * gridDim.x, per_group = (unsigned)a.n_tiles * (unsigned)a.parts;
            const unsigned group = g / per_group, in_group = g - group * per_group, tile = in_group / (unsigned)a.parts;
            const int part = (int)(in_group - tile * (unsigned)a.parts);
            const int2 at = __ldg(reinterpret_cast<const int2*>(a.tiles + tile));
            const MiniBucket* b = a.buckets + at.x;
            const int words = __ldg(reinterpret_cast<const int*>(b) + lane), more_words = __ldg(reinterpret_cast<const int*>(b) + 32 + lane), first = word(words, 2), combos = word(words, 3) - first;
            const int nch = word(words, 4), n0 = (int)group * a.examples, ne = min(a.examples, a.N - n0), beg = combos * part / a.parts;
            cur = TileAt{word(words, 0), word(words, 1), nch * kMPlaneBytes, at.y, n0, ne, first + beg, (combos * (part + 1) / a.parts - beg) * ne};
            fetch_rec();
            const FillAt columns(cur.d, cur.raster_len, cur.c0, a.L, lane);
            fill_planes(a, columns, planes, [&](int c) { return c < 20 ? word(words, 12 + c) : word(more_words, c - 20); }, nch, n0, ne, warp, kMWarps, lane);
            __syncthreads();
        } else {
            if (!mbar_wait(full0 + 8u * (k & 1), (k >> 1) & 1)) return false;
            cur = s_tile[k & 1];
            fetch_rec();
        }
        const int cg = cur.c0 + 2 * lane, band = (int)((unsigned)cg / (unsigned)cur.d);
        c0 = cg - band * cur.d;
        c1 = c0 + 1 < cur.d ? c0 + 1 : 0;
        trow0 = band * kMRows;
        trow1 = c0 + 1 < cur.d ? trow0 : trow0 + kMRows;
        ok0 = cg < cur.raster_len;
        ok1 = cg + 1 < cur.raster_len;
        return true;
    };
    ok = enter();
    while (ok) {
        if (pos >= base + cur.n_work) {
            if (k + 1 >= K) break;
            if constexpr (WIDE) {
                __syncthreads();
            } else {
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8u * (k & 1));
            }
            base += cur.n_work;
            ++k;
            ok = enter();
            continue;
        }
        const int rec = rec_next, w = pos - base, e = cur.ne == 1 ? 0 : w % cur.ne;
        const int m = word(rec, 0), f0 = word(rec, 1), nf = word(rec, 2);
        float my_bias = lane < nf ? __ldg(a.bias + f0 + lane) : 0.0f;
        pos = draw();
        fetch_rec();
        const char* st = reinterpret_cast<const char*>(planes + (WIDE ? 0 : (k & 1) * kMPlanes * kMPlaneFloats) + 2 * lane);
        if (e > 0) st += e * cur.plane_bytes;

        // the sum of the combination's channels, in the order of its list
        u64 xs[kMInRows];
        {
            const u64* p = reinterpret_cast<const u64*>(st + word(rec, 8));
#pragma unroll
            for (int s = 0; s < kMInRows; ++s) xs[s] = p[s * (kWarpCols / 2)];
        }
        for (int q = 1; q < m; ++q) {
            const u64* p = reinterpret_cast<const u64*>(st + word(rec, 8 + q));
#pragma unroll
            for (int s = 0; s < kMInRows; ++s) xs[s] = add2(xs[s], p[s * (kWarpCols / 2)]);
        }
        u64 acc[kMRows];                               // -z
        {
            u64 wp[kLen];
#pragma unroll
            for (int j = 0; j < kLen; ++j) {
                const float v = __int_as_float(word(rec, 17 + j));
                wp[j] = pack2(v, v);
            }
#pragma unroll
            for (int s = 0; s < kMInRows; ++s)
#pragma unroll
                for (int j = 0; j < kLen; ++j) {
                    const int o = s - j;
                    if (o >= 0 && o < kMRows) {
                        if (j == 0) acc[o] = fma2_to(wp[0], xs[s], 0ull);
                        else fma2(acc[o], wp[j], xs[s]);
                    }
                }
        }
        // outputs that do not exist: +inf, which no bias exceeds
        {
            const int tl = word(rec, 3), th = word(rec, 4);
            if (!__all_sync(kFull, ok1 && trow0 >= tl && trow1 + kMRows <= th)) {
                const int rh = word(rec, 5);
                int lo, hi;
                valid_rows_tc(trow0, c0, tl, 0, th, rh, kMRows, ok0, lo, hi);
                const unsigned m0 = row_mask(lo, hi);
                valid_rows_tc(trow1, c1, tl, 0, th, rh, kMRows, ok1, lo, hi);
                const unsigned m1 = row_mask(lo, hi);
                const float inf = __int_as_float(0x7f800000);
#pragma unroll
                for (int o = 0; o < kMRows; ++o) {
                    float x, y;
                    unpack2(acc[o], x, y);
                    acc[o] = pack2((m0 >> o) & 1 ? x : inf, (m1 >> o) & 1 ? y : inf);
                }
            }
        }
        // Eq. 1 against every bias; two of them share a reduction over the warp, lane f keeps the count of bias f
        int* counts = a.counts + (size_t)(cur.n0 + e) * a.F + f0;
        for (int fb = 0; fb < nf; fb += 32) {
            if (fb > 0) my_bias = fb + lane < nf ? __ldg(a.bias + f0 + fb + lane) : 0.0f;
            const int n = min(32, nf - fb);
            int mine = 0;
            for (int f = 0; f < n; f += 2) {
                int both = mini_count(acc, __shfl_sync(kFull, my_bias, f));
                if (f + 1 < n) both |= mini_count(acc, __shfl_sync(kFull, my_bias, f + 1)) << 16;
                both = __reduce_add_sync(kFull, both);
                if ((lane & ~1) == f) mine = lane & 1 ? both >> 16 : both & 0xffff;
            }
            if (lane < n && mine) atomicAdd(counts + fb + lane, mine);
        }
    }
    if (!ok && lane == 0) atomicExch(a.failed, 1);
}

// A call's flag, set when one of its waits gave up, and the blocks of its finalising kernel that have read it then.
struct MiniFlag { int failed; unsigned readers; };
constexpr int kMFlags = 64;               // calls take them in turn

// Counts to shares of outputs (Eq. 2); NaN when a wait of the tile kernel gave up, in which case the last block clears the flag, so
// that the failure stays the call's own (also where a graph repeats the call).
__global__ void __launch_bounds__(256)
mini_finalize_kernel(float* __restrict__ feat, const int* __restrict__ nout, int F, long long total, MiniFlag* flag) {
    dependency_wait();
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    const bool failed = *(volatile int*)&flag->failed != 0;
    if (i < total) {
        const int count = reinterpret_cast<const int*>(feat)[i];
        feat[i] = failed ? __int_as_float(0x7fc00000) : (float)count / (float)__ldg(nout + i % F);
    }
    if (!failed) return;
    __syncthreads();                      // every thread of the block has read the flag
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&flag->readers, 1u) == gridDim.x - 1) {
            flag->readers = 0u;
            flag->failed = 0;
        }
    }
}

}  // namespace
}  // namespace fast
}  // namespace rocket

using namespace rocket::fast;

struct rocket_mini {
    int C = 0, L = 0, F = 0, n_combos = 0;
    std::vector<int32_t> taps, dilation, kernel_index, padded, num_channels, channel_idx, channel_offset, feature_offset;
    std::vector<double> example_draw, quantile;
    std::vector<float> bias;
    bool fitted = false;
    std::vector<MiniRec> recs;
    std::vector<MiniBucket> buckets;
    std::vector<MiniTile> tiles;
    std::vector<WalkItem> walk_items;
    // what mini_walks compares, in us: copies and work of all tiles of one example; all walks of one example and the longest walk
    double us_copies = 0.0, us_work = 0.0, us_walks = 0.0, us_walk = 0.0;
    std::vector<int32_t> nout;             // outputs behind every feature
    int64_t slices = 0;                    // slices of at most eight features of one combination
    int max_nch = 1;
    bool wide = false;                     // the combinations of some dilation use more than kMPlanes channels
    mutable std::mutex mu;
    mutable int device = -1;
    mutable void* blob = nullptr;          // records, buckets, tiles, output counts, biases, the calls' flags
    mutable MiniArgs dev{};
    mutable const int* d_nout = nullptr;
    mutable const WalkItem* d_walk = nullptr;
    mutable MiniFlag* flags = nullptr;
    mutable std::atomic<unsigned> calls{0};
    mutable bool bias_uploaded = false;
};

// Groups the combinations of every dilation into buckets of at most kMPlanes channels and cuts their rasters into tiles.
static void build_tiles(rocket_mini& p) {
    p.recs.clear(); p.buckets.clear(); p.tiles.clear();
    p.nout.assign(p.F, 1);
    p.slices = 0;
    for (int c = 0; c < p.n_combos; ++c) p.slices += (p.feature_offset[c + 1] - p.feature_offset[c] + 7) / 8;
    p.max_nch = 1;
    std::map<int, std::vector<int>> by_d;
    for (int c = 0; c < p.n_combos; ++c)
        if (p.feature_offset[c + 1] > p.feature_offset[c]) by_d[p.dilation[c]].push_back(c);
    // A handle whose dilations all fit has two tiles in shared memory.  With more channels one large tile is better than several
    // small buckets for each dilation, which repeat channels and leave a tile only a dozen combinations.
    p.wide = false;
    for (const auto& kv : by_d) {
        std::vector<char> has(p.C, 0);
        for (int c : kv.second)
            for (int q = p.channel_offset[c]; q < p.channel_offset[c + 1]; ++q) has[p.channel_idx[q]] = 1;
        p.wide = p.wide || std::count(has.begin(), has.end(), 1) > kMPlanes;
    }
    const int planes = p.wide ? kMPlanesWide : kMPlanes;
    struct Group { std::vector<char> has; int nch; std::vector<int> combos; };
    for (auto& kv : by_d) {
        const int d = kv.first;
        auto& cs = kv.second;
        // most channels first: they find room while the groups are empty, and the long ones start first in a tile
        std::stable_sort(cs.begin(), cs.end(), [&](int a, int b) { return p.num_channels[a] > p.num_channels[b]; });
        std::vector<Group> groups;
        for (int c : cs) {
            const int32_t* S = p.channel_idx.data() + p.channel_offset[c];
            const int m = p.num_channels[c];
            int best = -1, best_new = 1 << 30;
            for (size_t g = 0; g < groups.size(); ++g) {
                int fresh = 0;
                for (int q = 0; q < m; ++q) fresh += !groups[g].has[S[q]];
                if (groups[g].nch + fresh <= planes && fresh < best_new) { best = (int)g; best_new = fresh; }
            }
            if (best < 0) { best = (int)groups.size(); groups.push_back({std::vector<char>(p.C, 0), 0, {}}); }
            Group& g = groups[best];
            for (int q = 0; q < m; ++q)
                if (!g.has[S[q]]) { g.has[S[q]] = 1; ++g.nch; }
            g.combos.push_back(c);
        }
        const int rows = (int)(((int64_t)p.L + d - 1) / d), bands = (rows + kMRows - 1) / kMRows;
        for (Group& g : groups) {
            MiniBucket b{};
            b.d = d; b.raster_len = bands * d;
            b.kbeg = (int)p.recs.size();
            std::vector<int> at(p.C, 0);
            for (int c = 0; c < p.C; ++c)
                if (g.has[c]) { b.ch[b.nch] = c; at[c] = b.nch++; }
            p.max_nch = std::max(p.max_nch, b.nch);
            for (int c : g.combos) {
                MiniRec r{};
                r.m = p.num_channels[c];
                for (int j = 0; j < kLen; ++j) r.w[j] = 1.0f;
                for (int t = 0; t < 3; ++t) r.w[p.taps[3 * p.kernel_index[c] + t]] = -2.0f;
                r.f0 = p.feature_offset[c]; r.nf = p.feature_offset[c + 1] - r.f0;
                const int first = p.padded[c] ? 0 : 4 * d, last = p.padded[c] ? p.L : p.L - 4 * d;
                r.tl = first / d; r.th = last / d; r.rh = last - r.th * d;
                for (int q = 0; q < r.m; ++q) r.ch[q] = at[p.channel_idx[p.channel_offset[c] + q]] * kMPlaneBytes;
                for (int f = r.f0; f < r.f0 + r.nf; ++f) p.nout[f] = last - first;
                p.recs.push_back(r);
            }
            b.kend = (int)p.recs.size();
            for (int c0 = 0; c0 < b.raster_len; c0 += kWarpCols) p.tiles.push_back({(int)p.buckets.size(), c0});
            p.buckets.push_back(b);
        }
    }
}

// Costs for mini_walks, fitted to the device times of 600 calls of 1 to 250 channels, 24 to 60,000 steps, 84 to 9,996 features and 1 to
// 128 examples (13 % rms for the walks, 25 % for the tiles, which have costs of their own where a dilation is several buckets).
struct TileCosts { double call, tile, plane, pair, channel, bias, tie; };      // tie: the tiles have it within this
constexpr TileCosts kUsOneBucket{6.75, 4.68, 0.092, 0.0673, 0.0176, 0.0131, 1.1}, kUsBuckets{6.81, 7.81, 0.0, 0.179, 0.0, 0.0023, 1.02};
constexpr double kUsWalks = 2.86, kUsItem = 1.17, kUsLoad = 5.1e-5, kUsStaged = 1.13e-4, kUsLongest = 2.69e-4;
static const TileCosts& tile_costs(const rocket_mini& p) { return p.C > kMPlanesWide ? kUsBuckets : kUsOneBucket; }

// The items of the kernel that takes one combination at a time, and the costs of either kernel.
static void build_walk_items(rocket_mini& p) {
    p.us_copies = p.us_work = p.us_walks = p.us_walk = 0.0;
    const TileCosts& us = tile_costs(p);
    std::vector<double> work(p.buckets.size(), 0.0);
    for (size_t b = 0; b < p.buckets.size(); ++b)
        for (int r = p.buckets[b].kbeg; r < p.buckets[b].kend; ++r) work[b] += us.pair + p.recs[r].m * us.channel + p.recs[r].nf * us.bias;
    for (const MiniTile& t : p.tiles) {
        p.us_copies += us.plane * p.buckets[t.bucket].nch;
        p.us_work += work[t.bucket];
    }
    p.walk_items.clear();
    if (p.L > kWalkMostSamples) return;
    struct Tiling { int width, seg_rows, segs; double staged, slots; };
    std::map<int, Tiling> tiling;                        // by dilation
    for (int c = 0; c < p.n_combos; ++c)
        for (int f0 = p.feature_offset[c]; f0 < p.feature_offset[c + 1]; f0 += kWalkFeatures) {
            WalkItem it{};
            it.d = p.dilation[c]; it.padded = p.padded[c]; it.m = p.num_channels[c];
            it.f0 = f0; it.nf = std::min(kWalkFeatures, p.feature_offset[c + 1] - f0);
            for (int k = 0; k < 3; ++k) it.tap[k] = p.taps[3 * p.kernel_index[c] + k];
            for (int q = 0; q < it.m; ++q) it.ch[q] = p.channel_idx[p.channel_offset[c] + q];
            auto found = tiling.find(it.d);
            if (found == tiling.end()) {
                Tiling t{};
                choose_walk(it.d, p.L, t.width, t.seg_rows, t.segs);
                if (t.width < 1 || t.seg_rows < kLen || t.segs < 1 || (int64_t)(t.seg_rows * t.segs + 8) * t.width > kWalkSamples) {
                    p.walk_items.clear();                // no tiling fits (does not happen from L = 9 on)
                    return;
                }
                const int T = (p.L + it.d - 1) / it.d, tile_rows = t.seg_rows * t.segs;
                for (int ta = 0; ta < T; ta += tile_rows) {
                    const int rows = std::min(tile_rows, T - ta), segs = (rows + t.seg_rows - 1) / t.seg_rows;
                    for (int ca = 0; ca < it.d; ca += t.width) {
                        const int cols = std::min(t.width, it.d - ca);
                        t.staged += (rows + 8.0) * cols;
                        t.slots += (double)(((int64_t)cols * segs + kWalkThreads - 1) / kWalkThreads * kWalkThreads) * (std::min(t.seg_rows, rows) + 1);
                    }
                }
                found = tiling.emplace(it.d, t).first;
            }
            const Tiling& t = found->second;
            it.width = t.width; it.seg_rows = t.seg_rows; it.segs = t.segs;
            p.walk_items.push_back(it);
            p.us_walks += kUsItem + t.staged * it.m * kUsLoad + t.staged * kUsStaged;
            p.us_walk = std::max(p.us_walk, kUsLongest * (0.3 * t.staged * it.m + t.slots));
        }
}

// How the tile kernel goes over N examples.
struct MiniLaunch { int examples, groups, parts; unsigned grid; bool all_copy; };
static MiniLaunch mini_launch(const rocket_mini& p, int N, int sms) {
    MiniLaunch a;
    // Examples that share a tile: as many as its planes hold, while every SM still gets four tiles; fewer tiles than SMs are
    // dealt in parts of their combinations (84 or so) instead.
    const long long n_tiles = (long long)p.tiles.size(), tiles = N * n_tiles;
    a.examples = (int)std::max<long long>(1, std::min<long long>({(p.wide ? kMPlanesWide : kMPlanes) / p.max_nch, N, tiles / (4ll * sms)}));
    a.groups = (N + a.examples - 1) / a.examples;
    const long long items = (long long)a.groups * n_tiles;
    a.parts = (int)std::max<long long>(1, std::min<long long>(8, 2ll * sms / items));
    a.grid = (unsigned)std::min<long long>(items * a.parts, sms);
    // A block that has one tile only has nothing to overlap its copies with: all warps make them (1 x 20 x 300, 840 features:
    // 16.4 us with three warps, 14.4 so), into no more shared memory than the tile takes (1 x 12 x 900: 16.4 -> 14.4 us).
    a.all_copy = p.wide || items * a.parts <= a.grid;
    return a;
}

// Whether the kernel that takes one combination at a time serves a call of N examples in less time.  It does where a tile's channels are
// many and each is used by few combinations (24 x 250 x 10,000, 9,996 features: 1.65 ms against 4.5; 24 x 100 x 10,000, 840: 0.56
// against 1.35), and where there are few tiles (5 x 20 x 10,000, 84 features: 18.6 us against 26.7; 1 x 20 x 1,500, 840: 16 against
// 25).  The tiles have it from a few examples on where they share (24 x 20 x 10,000, 9,996 features: 0.88 ms against 1.6).
static bool mini_walks(const rocket_mini& p, int N, int sms) {
    if (p.walk_items.empty()) return false;
    const MiniLaunch a = mini_launch(p, N, sms);
    const double n_tiles = (double)p.tiles.size(), items = (double)a.groups * n_tiles * a.parts;
    auto both = [](double x, double y) { return std::sqrt(std::sqrt(x * x * x * x + y * y * y * y)); };   // near the larger
    const TileCosts& us = tile_costs(p);
    const double copies = us.tile + p.us_copies / n_tiles * a.examples, work = p.us_work / n_tiles * a.examples / a.parts;
    const double rounds = items / a.grid, tiles = us.call + (rounds < 4.0 ? std::ceil(rounds) : rounds + 0.5) * (a.all_copy ? copies + work : both(copies, work));
    return us.tie * (kUsWalks + both(N * p.us_walks / sms, p.us_walk)) < tiles;
}

// Examples of one launch of the tile kernel: (tile, example) pairs, eight parts of each, are counted in 32 bits.
#ifndef ROCKET_MINI_LAUNCH_TILES
#define ROCKET_MINI_LAUNCH_TILES (0x7fffffffll / 8)
#endif
static int mini_launch_examples(long long n_tiles) { return (int)std::max<long long>(1, std::min<long long>(0x7fffffff, ROCKET_MINI_LAUNCH_TILES / n_tiles)); }

static constexpr size_t kMiniSmemBytes = (size_t)2 * kMPlanes * kMPlaneBytes;

static int ensure_mini_device(const rocket_mini* p) {
    std::lock_guard<std::mutex> lk(p->mu);
    if (p->device < 0) {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
        struct Part { const void* src; size_t bytes, off; };
        Part parts[7] = {{p->recs.data(), p->recs.size() * sizeof(MiniRec), 0},     {p->buckets.data(), p->buckets.size() * sizeof(MiniBucket), 0},
                         {p->tiles.data(), p->tiles.size() * sizeof(MiniTile), 0}, {p->nout.data(), p->nout.size() * sizeof(int32_t), 0},
                         {nullptr, (size_t)p->F * sizeof(float), 0},               {nullptr, kMFlags * sizeof(MiniFlag), 0},
                         {p->walk_items.data(), p->walk_items.size() * sizeof(WalkItem), 0}};
        size_t total = 0;
        for (Part& pt : parts) { pt.off = total; total += (pt.bytes + 255) / 256 * 256; }
        cudaError_t e = rocket::device_malloc(&p->blob, total);
        if (e != cudaSuccess) { cudaGetLastError(); p->blob = nullptr; return e == cudaErrorMemoryAllocation ? ROCKET_ENOMEM : ROCKET_ECUDA; }
        char* base = static_cast<char*>(p->blob);
        e = cudaMemset(base + parts[5].off, 0, parts[5].bytes);
        for (const Part& pt : parts)
            if (e == cudaSuccess && pt.src && pt.bytes) e = cudaMemcpy(base + pt.off, pt.src, pt.bytes, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(mini_tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMiniSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(mini_tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMiniSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(mini_walk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kWalkSamples * sizeof(float)));
        if (e != cudaSuccess) { cudaGetLastError(); cudaFree(p->blob); p->blob = nullptr; return ROCKET_ECUDA; }
        MiniArgs& a = p->dev;
        a.recs = reinterpret_cast<const MiniRec*>(base + parts[0].off);
        a.buckets = reinterpret_cast<const MiniBucket*>(base + parts[1].off);
        a.tiles = reinterpret_cast<const MiniTile*>(base + parts[2].off);
        p->d_nout = reinterpret_cast<const int*>(base + parts[3].off);
        a.bias = reinterpret_cast<const float*>(base + parts[4].off);
        p->d_walk = reinterpret_cast<const WalkItem*>(base + parts[6].off);
        p->flags = reinterpret_cast<MiniFlag*>(base + parts[5].off);
        a.C = p->C; a.L = p->L; a.F = p->F; a.n_tiles = (int)p->tiles.size();
        p->device = dev;
        p->bias_uploaded = false;
    }
    if (!p->bias_uploaded) {
        int prev = -1;
        cudaGetDevice(&prev);
        if (prev != p->device) cudaSetDevice(p->device);
        const cudaError_t e = cudaMemcpy(const_cast<float*>(p->dev.bias), p->bias.data(), (size_t)p->F * sizeof(float), cudaMemcpyHostToDevice);
        if (prev != p->device) cudaSetDevice(prev);
        if (e != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
        p->bias_uploaded = true;
    }
    return ROCKET_OK;
}

extern "C" {

int rocket_mini_create(uint64_t seed, int C, int L, int num_features, rocket_mini_t** out) {
    if (!out || C < 1 || L < kLen || num_features < kKernels) return ROCKET_EINVAL;
    if ((int64_t)C * L > 0x7fffffffll) return ROCKET_EUNSUPPORTED;     // positions within an example are 32-bit
    rocket_mini* p = new (std::nothrow) rocket_mini();
    if (!p) return ROCKET_ENOMEM;
    try {
        p->C = C; p->L = L; p->F = (num_features / kKernels) * kKernels;
        for (int a = 0; a < kLen; ++a)
            for (int b = a + 1; b < kLen; ++b)
                for (int c = b + 1; c < kLen; ++c) { p->taps.push_back(a); p->taps.push_back(b); p->taps.push_back(c); }
        // dilations and the share of every kernel's features each of them holds
        const int fpk = p->F / kKernels, n = std::min(fpk, 32);
        const double E = std::log2((L - 1.0) / 8.0);
        std::vector<int64_t> dil;
        std::vector<int64_t> count;
        for (int k = 0; k < n; ++k) {
            const double x = n > 1 ? k * E / (n - 1) : 0.0;
            // a power that is an integer (the last one is (L - 1) / 8) must not fall below it by exp2's rounding
            const int64_t d = (int64_t)std::floor(std::exp2(x) * (1.0 + 0x1.0p-40));
            if (!dil.empty() && dil.back() == d) ++count.back();
            else { dil.push_back(d); count.push_back(1); }
        }
        std::vector<int> share(dil.size());
        int left = fpk;
        for (size_t i = 0; i < dil.size(); ++i) { share[i] = (int)std::floor(count[i] * ((double)fpk / n)); left -= share[i]; }
        for (size_t i = 0; left > 0; i = (i + 1) % dil.size()) { ++share[i]; --left; }
        p->n_combos = (int)dil.size() * kKernels;
        p->channel_offset.assign(1, 0);
        p->feature_offset.assign(1, 0);
        const int cap = std::min(C, kLen);
        std::vector<uint64_t> keys(C);
        std::vector<int> order(C);
        for (int c = 0; c < p->n_combos; ++c) {
            const int i_d = c / kKernels, kappa = c % kKernels;
            const uint64_t stream = (uint64_t)c + kStreamBase;
            int m = (int)std::floor(std::exp2(draw_uniform(seed, stream, 0) * std::log2(cap + 1.0)));
            m = std::max(1, std::min(m, cap));
            for (int ch = 0; ch < C; ++ch) keys[ch] = draw_u64(seed, stream, 1024 + (uint64_t)ch);
            std::iota(order.begin(), order.end(), 0);
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return keys[a] < keys[b]; });
            std::vector<int> chosen(order.begin(), order.begin() + m);
            std::sort(chosen.begin(), chosen.end());
            for (int ch : chosen) p->channel_idx.push_back(ch);
            p->dilation.push_back((int32_t)dil[i_d]); p->kernel_index.push_back(kappa);
            p->padded.push_back((i_d + kappa) % 2 == 0 ? 1 : 0); p->num_channels.push_back(m);
            p->channel_offset.push_back((int32_t)p->channel_idx.size());
            p->feature_offset.push_back(p->feature_offset.back() + share[i_d]);
            p->example_draw.push_back(draw_uniform(seed, stream, 1));
        }
        p->quantile.resize(p->F);
        for (int f = 0; f < p->F; ++f) p->quantile[f] = std::fmod((f + 1.0) * kInvGoldenRatio, 1.0);
        p->bias.assign(p->F, 0.0f);
        build_tiles(*p);
        build_walk_items(*p);
    } catch (const std::bad_alloc&) {
        delete p;
        return ROCKET_ENOMEM;
    }
    *out = p;
    return ROCKET_OK;
}

int rocket_mini_counts(const rocket_mini_t* p, int* C, int* L, int* n_features, int* n_combinations, int64_t* n_channel_idx) {
    if (!p) return ROCKET_EINVAL;
    if (C) *C = p->C;
    if (L) *L = p->L;
    if (n_features) *n_features = p->F;
    if (n_combinations) *n_combinations = p->n_combos;
    if (n_channel_idx) *n_channel_idx = (int64_t)p->channel_idx.size();
    return ROCKET_OK;
}

int rocket_mini_host_view(const rocket_mini_t* p, const int32_t** taps, const int32_t** dilation, const int32_t** kernel_index,
                          const int32_t** padded, const int32_t** num_channels, const int32_t** channel_idx,
                          const int32_t** feature_offset, const double** example_draw, const double** quantile,
                          const float** bias) {
    if (!p) return ROCKET_EINVAL;
    if (taps) *taps = p->taps.data();
    if (dilation) *dilation = p->dilation.data();
    if (kernel_index) *kernel_index = p->kernel_index.data();
    if (padded) *padded = p->padded.data();
    if (num_channels) *num_channels = p->num_channels.data();
    if (channel_idx) *channel_idx = p->channel_idx.data();
    if (feature_offset) *feature_offset = p->feature_offset.data();
    if (example_draw) *example_draw = p->example_draw.data();
    if (quantile) *quantile = p->quantile.data();
    if (bias) *bias = p->bias.data();
    return ROCKET_OK;
}

int rocket_mini_fit(rocket_mini_t* p, const float* X_host, int N) {
    if (!p || !X_host || N < 1) return ROCKET_EINVAL;
    const int L = p->L, C = p->C;
    std::vector<float> bias(p->F);
    const unsigned hw = std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
    std::vector<std::thread> pool;
    std::atomic<int> next{0};
    std::atomic<bool> failed{false};
    auto worker = [&]() {
        try {
            std::vector<double> xs(L), z;
            for (int c = next.fetch_add(1); c < p->n_combos; c = next.fetch_add(1)) {
                const int n = std::min((int)(p->example_draw[c] * N), N - 1);
                const float* Xn = X_host + (size_t)n * C * L;
                const int d = p->dilation[c];
                std::fill(xs.begin(), xs.end(), 0.0);
                for (int q = p->channel_offset[c]; q < p->channel_offset[c + 1]; ++q) {
                    const float* x = Xn + (size_t)p->channel_idx[q] * L;
                    for (int i = 0; i < L; ++i) xs[i] += (double)x[i];
                }
                const int32_t* tap = p->taps.data() + 3 * p->kernel_index[c];
                const int first = p->padded[c] ? 0 : 4 * d, last = p->padded[c] ? L : L - 4 * d;
                z.resize(last - first);
                for (int i = first; i < last; ++i) {
                    double v = 0.0;
                    for (int j = 0; j < kLen; ++j) {
                        const long long t = (long long)i + (long long)(j - 4) * d;
                        if (t >= 0 && t < L) v += ((j == tap[0] || j == tap[1] || j == tap[2]) ? 2.0 : -1.0) * xs[t];
                    }
                    z[i - first] = v;
                }
                std::sort(z.begin(), z.end());
                const long long nz = (long long)z.size();
                for (int f = p->feature_offset[c]; f < p->feature_offset[c + 1]; ++f) {
                    const double pos = p->quantile[f] * (double)(nz - 1);
                    const long long lo = (long long)std::floor(pos), hi = std::min(lo + 1, nz - 1);
                    bias[f] = (float)(z[lo] + (pos - (double)lo) * (z[hi] - z[lo]));
                }
            }
        } catch (...) {
            failed = true;
        }
    };
    try {
        for (unsigned t = 0; t < hw; ++t) pool.emplace_back(worker);
    } catch (...) {
        failed = failed || pool.empty();
    }
    for (auto& t : pool) t.join();
    if (failed) return ROCKET_ENOMEM;
    std::lock_guard<std::mutex> lk(p->mu);
    p->bias.swap(bias);
    p->fitted = true;
    p->bias_uploaded = false;
    return ROCKET_OK;
}

int rocket_mini_set_biases(rocket_mini_t* p, const float* bias) {
    if (!p || !bias) return ROCKET_EINVAL;
    for (int f = 0; f < p->F; ++f)
        if (!(bias[f] - bias[f] == 0.0f)) return ROCKET_EINVAL;
    std::lock_guard<std::mutex> lk(p->mu);
    p->bias.assign(bias, bias + p->F);
    p->fitted = true;
    p->bias_uploaded = false;
    return ROCKET_OK;
}

int rocket_mini_transform(const rocket_mini_t* p, const float* X_dev, int N, int C, int L, float* feat_dev, void* cuda_stream) {
    if (!p || N < 0) return ROCKET_EINVAL;
    if (C != p->C || L != p->L) return ROCKET_ESHAPE;
    if (!p->fitted) return ROCKET_EINVAL;
    if (N == 0) return ROCKET_OK;
    if (!X_dev || !feat_dev) return ROCKET_EINVAL;
    if (N * p->slices > 0x7fffffffll) return ROCKET_EUNSUPPORTED;
    const int st = ensure_mini_device(p);
    if (st != ROCKET_OK) return st;
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
    if (prev != p->device && cudaSetDevice(p->device) != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
    int sms = 0;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
    sms = std::max(sms, 1);
    if (mini_walks(*p, N, sms)) {
        mini_walk_kernel<<<(unsigned)(N * (long long)p->walk_items.size()), kWalkThreads, kWalkSamples * sizeof(float), stream>>>(
            X_dev, C, L, p->d_walk, (int)p->walk_items.size(), p->dev.bias, feat_dev, p->F);
        rocket::count_launch();
        const cudaError_t e = cudaGetLastError();
        if (prev != p->device) cudaSetDevice(prev);
        if (e != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
        return ROCKET_OK;
    }
    MiniFlag* flag = p->flags + p->calls.fetch_add(1, std::memory_order_relaxed) % kMFlags;
    const long long values = (long long)N * p->F;
    const unsigned value_blocks = (unsigned)((values + 255) / 256);
    cudaMemsetAsync(feat_dev, 0, (size_t)values * sizeof(float), stream);
    const int most = mini_launch_examples(p->dev.n_tiles);
    for (int n0 = 0; n0 < N; n0 += std::min(most, N - n0)) {
        MiniArgs args = p->dev;
        args.X = X_dev + (size_t)n0 * C * L;
        args.counts = reinterpret_cast<int*>(feat_dev) + (size_t)n0 * p->F;
        args.N = std::min(most, N - n0);
        args.failed = &flag->failed;
        const MiniLaunch at = mini_launch(*p, args.N, sms);
        args.examples = at.examples;
        args.groups = at.groups;
        args.parts = at.parts;
        if (at.all_copy) mini_tile_kernel<true><<<at.grid, kMThreads, (size_t)args.examples * p->max_nch * kMPlaneBytes, stream>>>(args);
        else mini_tile_kernel<false><<<at.grid, kMThreads, kMiniSmemBytes, stream>>>(args);
        rocket::count_launch();
    }
    launch_dependent(mini_finalize_kernel, value_blocks, 256, 0, stream, feat_dev, p->d_nout, p->F, values, flag);
    rocket::count_launch();
    const cudaError_t e = cudaGetLastError();
    if (prev != p->device) cudaSetDevice(prev);
    if (e != cudaSuccess) { cudaGetLastError(); return ROCKET_ECUDA; }
    return ROCKET_OK;
}

void rocket_mini_destroy(rocket_mini_t* p) {
    if (!p) return;
    if (p->device >= 0 && p->blob) {
        int prev = -1;
        cudaGetDevice(&prev);
        if (prev != p->device) cudaSetDevice(p->device);
        cudaFree(p->blob);
        if (prev >= 0 && prev != p->device) cudaSetDevice(prev);
        cudaGetLastError();
    }
    delete p;
}

}  // extern "C"
