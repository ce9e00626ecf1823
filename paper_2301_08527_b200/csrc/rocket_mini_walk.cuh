// MINIROCKET, a block per (example, combination): the form for little to share between the combinations of a tile.
//
// A block stages the channel-summed tile of one combination and its threads walk down the columns; a call is one launch.  Bound: the
// traffic from L2, every combination reads its channels once.  Against the kernel that shares a tile of all channels among the
// combinations of a dilation (rocket_mini.cu) it wins where there are many channels, of which a combination uses four on
// average, or too few tiles for the SMs: see mini_walks.
#pragma once

#include <climits>
#include <cstdint>
#include <type_traits>

#include "rocket_fast_dev.cuh"

namespace rocket {
namespace fast {
namespace {

constexpr int kWalkLen = 9;
constexpr int kWalkFeatures = 8;            // a combination with more features becomes several items
constexpr int kWalkThreads = 256, kWalkBlocks = 3;
constexpr int kWalkMostSamples = 1 << 28;   // a longer series has eight channels at most, which are better shared
constexpr int kWalkSamples = 16 * 1024;     // channel-summed samples a block stages at a time (64 KB of shared memory)

// One unit of work: a combination, or a slice of at most 8 of its features, with the tiling of the dilated view that the kernel uses
// for its dilation (chosen on the host, choose_walk).
struct WalkItem {
    int32_t d, padded, m, f0, nf;
    int32_t tap[3];
    int32_t ch[kWalkLen];
    int32_t width, seg_rows, segs;   // columns of a tile (= its pitch), rows a thread walks, such runs per tile
};
static_assert(sizeof(WalkItem) == 80, "WalkItem layout");

// Sample k of a channel row through the read-only path: at a constant byte offset from the row's first sample
// (STRIDE samples apart), or, with a run-time stride, at an address formed by one widening multiply-add.
template <int STRIDE>
__device__ __forceinline__ float load_at(const float* __restrict__ x0, int k, int stride) {
    float v;
    if constexpr (STRIDE != 0) {
        switch (k) {   // k is a constant after unrolling; the offset must be an immediate
            case 0: asm("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(x0)); break;
            case 1: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(4 * STRIDE)); break;
            case 2: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(8 * STRIDE)); break;
            case 3: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(12 * STRIDE)); break;
            case 4: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(16 * STRIDE)); break;
            case 5: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(20 * STRIDE)); break;
            case 6: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(24 * STRIDE)); break;
            default: asm("ld.global.nc.f32 %0, [%1+%2];" : "=f"(v) : "l"(x0), "n"(28 * STRIDE)); break;
        }
    } else {
        const float* p;
        asm("mad.wide.s32 %0, %1, 4, %2;" : "=l"(p) : "r"(k * stride), "l"(x0));
        asm("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    }
    return v;
}

// One output of the convolution from the nine window entries (the oldest sits in slot S0; taps are taken in
// the order 0..8 whatever the slot), compared with the first 4 NG biases of the item (Eq. 1 against the bias).
template <int S0, int NG>
__device__ __forceinline__ void walk_pool(const float (&win)[kWalkLen], const float (&w)[kWalkLen],
                                          const float (&b)[kWalkFeatures], int (&cnt)[kWalkFeatures]) {
    float z = 0.0f;
#pragma unroll
    for (int j = 0; j < kWalkLen; ++j) z = fmaf(w[j], win[(S0 + j) % kWalkLen], z);
    // Eq. 1 against every bias: one compare and one predicated add each
#pragma unroll
    for (int f = 0; f < 4 * NG; ++f)
        asm("{ .reg .pred p; setp.gt.f32 p, %1, %2; @p add.s32 %0, %0, 1; }" : "+r"(cnt[f]) : "f"(z), "f"(b[f]));
}

// Steps K .. 8 of a group of nine outputs: the next row's sample enters the slot the oldest one leaves, so
// the window never moves between registers.  GUARD: the run may end inside the group.
template <int K, bool GUARD, int NG>
__device__ __forceinline__ void walk_steps(const float*& p, int pitch, int left, float (&win)[kWalkLen], const float (&w)[kWalkLen],
                                           const float (&b)[kWalkFeatures], int (&cnt)[kWalkFeatures]) {
    if constexpr (K < kWalkLen) {
        if (!GUARD || K < left) {
            win[(K + kWalkLen - 1) % kWalkLen] = *p;
            p += pitch;
            walk_pool<K, NG>(win, w, b, cnt);
        }
        walk_steps<K + 1, GUARD, NG>(p, pitch, left, win, w, b, cnt);
    }
}

// The walks over one staged tile: thread u of cols * segs takes column u % cols over run u / cols.  Outputs of
// column c are the rows t_min <= t < t_full + (c < c_more): t d + c < last with last = t_full d + c_more.
template <int NG>
__device__ __forceinline__ void walk_tile(const float* s_x, int P, int cols, int rows, int seg_rows, int ta, int ca,
                                               int t_min, int t_full, int c_more, const float (&w)[kWalkLen],
                                               const float (&b)[kWalkFeatures], int (&cnt)[kWalkFeatures]) {
    const int segs = (rows + seg_rows - 1) / seg_rows;
    // (run, column) of thread u, stepped without divisions: u advances by the block's threads
    const int dq = kWalkThreads / cols, dr = kWalkThreads - dq * cols;
    int seg = threadIdx.x / cols, c = threadIdx.x - seg * cols;
    for (int u = threadIdx.x; u < cols * segs; u += kWalkThreads) {
        const int t_end = t_full + (ca + c < c_more ? 1 : 0);
        const int t_lo = max(ta + seg * seg_rows, t_min);
        const int t_hi = min(min(ta + rows, ta + (seg + 1) * seg_rows), t_end);
        int left = t_hi - t_lo;
        if (left > 0) {
            // the window of output row t holds rows t - 4 .. t + 4; staged row 0 is row ta - 4
            const float* p = s_x + (t_lo - ta) * P + c;
            float win[kWalkLen];
#pragma unroll
            for (int j = 0; j < kWalkLen - 1; ++j) { win[j] = *p; p += P; }
            for (; left >= kWalkLen; left -= kWalkLen) walk_steps<0, false, NG>(p, P, left, win, w, b, cnt);
            if (left > 0) walk_steps<0, true, NG>(p, P, left, win, w, b, cnt);
        }
        seg += dq; c += dr;
        if (c >= cols) { c -= cols; ++seg; }
    }
}

// One block per (example, item).  The series is seen as rows of d samples (A[t][c] = x[t d + c]); a tile of it -
// rows [ta - 4, ta + rows + 4) of `width` columns, channels already summed, zeros outside the series - is
// staged in shared memory, then every thread walks down one column over a run of seg_rows rows with the nine
// taps in registers: one shared-memory load, nine multiply-adds and the bias compares per output.
__global__ void __launch_bounds__(kWalkThreads, kWalkBlocks)
mini_walk_kernel(const float* __restrict__ X, int C, int L, const WalkItem* __restrict__ items, int n_items,
                      const float* __restrict__ bias, float* __restrict__ feat, int F) {
    extern __shared__ float s_x[];
    __shared__ int s_cnt[kWalkFeatures];
    __shared__ int s_choff[kWalkLen];
    const int n = blockIdx.x / n_items;
    const WalkItem* __restrict__ item = items + (blockIdx.x - n * n_items);
    const WalkItem it = *item;
    const float* __restrict__ Xn = X + (size_t)n * C * L;
    const int tid = threadIdx.x;
    if (tid < kWalkFeatures) s_cnt[tid] = 0;
    if (tid < kWalkLen) s_choff[tid] = __ldg(item->ch + (tid < it.m ? tid : 0)) * L;     // C L < 2^31 (checked at creation)
    const int d = it.d, m = it.m, nf = it.nf;
    const int first = it.padded ? 0 : 4 * d, last = it.padded ? L : L - 4 * d;
    float w[kWalkLen];
#pragma unroll
    for (int j = 0; j < kWalkLen; ++j) w[j] = (j == it.tap[0] || j == it.tap[1] || j == it.tap[2]) ? 2.0f : -1.0f;
    float b[kWalkFeatures];
#pragma unroll
    for (int f = 0; f < kWalkFeatures; ++f) b[f] = f < nf ? __ldg(bias + it.f0 + f) : __int_as_float(0x7f800000);
    int cnt[kWalkFeatures];
#pragma unroll
    for (int f = 0; f < kWalkFeatures; ++f) cnt[f] = 0;

    const int T = (L + d - 1) / d;                       // rows of the dilated view
    const int P = it.width, seg_rows = it.seg_rows;      // P: columns of a tile and its pitch in shared memory
    const int tile_rows = seg_rows * it.segs;
    const bool whole_rows = P == d;                      // a tile spans whole rows: its samples are one contiguous run
    const int t_min = it.padded ? 0 : 4;                 // rows below hold no output of an unpadded combination
    const int t_full = last / d, c_more = last - t_full * d;   // column c has outputs in rows t < t_full + (c < c_more)
    const int groups = (nf + 3) / 4;

    // NK staged samples per thread at a time: position base + k * stride goes to slot + k * slot_stride.  The
    // channels are taken two at a time, so that 2 NK loads are in flight per thread.  CHECK: a sample may lie
    // beyond the series (then it is zero).  STRIDE = 0: the stride is a run-time value.
    auto stage = [&](auto nk_tag, auto stride_tag, auto check_tag, int base, int stride_rt, int slot, int slot_stride) {
        constexpr int NK = decltype(nk_tag)::value;
        constexpr int STRIDE = decltype(stride_tag)::value;
        constexpr bool CHECK = decltype(check_tag)::value;
        const int stride = STRIDE ? STRIDE : stride_rt;
        float acc[NK];
        bool ok[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            acc[k] = 0.0f;
            ok[k] = !CHECK || (unsigned)(base + k * stride) < (unsigned)L;
        }
        int q = 0;
        for (; q + 2 <= m; q += 2) {
            const float* __restrict__ x0 = Xn + s_choff[q] + base;
            const float* __restrict__ x1 = Xn + s_choff[q + 1] + base;
            float v0[NK], v1[NK];
#pragma unroll
            for (int k = 0; k < NK; ++k) {
                v0[k] = ok[k] ? load_at<STRIDE>(x0, k, stride) : 0.0f;
                v1[k] = ok[k] ? load_at<STRIDE>(x1, k, stride) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < NK; ++k) acc[k] = (acc[k] + v0[k]) + v1[k];
        }
        if (q < m) {
            const float* __restrict__ x0 = Xn + s_choff[q] + base;
#pragma unroll
            for (int k = 0; k < NK; ++k)
                if (ok[k]) acc[k] += load_at<STRIDE>(x0, k, stride);
        }
#pragma unroll
        for (int k = 0; k < NK; ++k) s_x[slot + k * slot_stride] = acc[k];
    };
    using Strided = std::integral_constant<int, 0>;
    using Dense = std::integral_constant<int, kWalkThreads>;
    using N8 = std::integral_constant<int, 8>;
    using N4 = std::integral_constant<int, 4>;
    using N2 = std::integral_constant<int, 2>;
    using N1 = std::integral_constant<int, 1>;
    using Checked = std::true_type;
    using Inside = std::false_type;

    for (int ta = 0; ta < T; ta += tile_rows) {
        const int rows = min(tile_rows, T - ta);
        for (int ca = 0; ca < d; ca += P) {
            const int cols = min(P, d - ca);
            __syncthreads();                             // the previous tile's walks are over (and s_choff is written)
            if (whole_rows) {
                // slots [0, count) hold positions g0 .. g0 + count: zeros before the series, the samples in
                // rounds of 8 x 256 and of 256 without any test, one last partial round, zeros after the series
                const int count = (rows + 8) * d, g0 = (ta - 4) * d;
                const int z0 = min(max(-g0, 0), count), z1 = min(max(L - g0, 0), count);
                for (int e = tid; e < z0; e += kWalkThreads) s_x[e] = 0.0f;
                for (int e = z1 + tid; e < count; e += kWalkThreads) s_x[e] = 0.0f;
                int e0 = z0;
                for (; e0 + 8 * kWalkThreads <= z1; e0 += 8 * kWalkThreads) stage(N8{}, Dense{}, Inside{}, g0 + e0 + tid, 0, e0 + tid, kWalkThreads);
                for (; e0 + kWalkThreads <= z1; e0 += kWalkThreads) stage(N1{}, Dense{}, Inside{}, g0 + e0 + tid, 0, e0 + tid, kWalkThreads);
                if (e0 + tid < z1) stage(N1{}, Dense{}, Inside{}, g0 + e0 + tid, 0, e0 + tid, kWalkThreads);
            } else {
                for (int cb = 0; cb < cols; cb += kWalkThreads) {
                    if (cb + tid >= cols) continue;
                    // staged row r is row ta - 4 + r of the view: zeros above the series, rows that lie inside it
                    // for every column of this block without any test, the rows the series ends in, zeros below
                    const int w = min(kWalkThreads, cols - cb), c_lo = ca + cb;
                    const int n_rows = rows + 8;
                    const int r_a = min(max(4 - ta, 0), n_rows);
                    const int t_full = L >= c_lo + w ? (L - c_lo - w) / d + 1 : 0;     // rows t < t_full hold all w columns
                    const int t_some = L > c_lo ? (L - c_lo - 1) / d + 1 : 0;          // rows t < t_some hold at least one
                    const int r_b = min(max(t_full - (ta - 4), r_a), n_rows), r_c = min(max(t_some - (ta - 4), r_b), n_rows);
                    const int pos0 = (ta - 4) * d + c_lo + tid, slot0 = cb + tid;
                    for (int r = 0; r < r_a; ++r) s_x[slot0 + r * P] = 0.0f;
                    int r = r_a;
                    for (; r + 8 <= r_b; r += 8) stage(N8{}, Strided{}, Inside{}, pos0 + r * d, d, slot0 + r * P, P);
                    if (r + 4 <= r_b) { stage(N4{}, Strided{}, Inside{}, pos0 + r * d, d, slot0 + r * P, P); r += 4; }
                    if (r + 2 <= r_b) { stage(N2{}, Strided{}, Inside{}, pos0 + r * d, d, slot0 + r * P, P); r += 2; }
                    if (r + 1 <= r_b) { stage(N1{}, Strided{}, Inside{}, pos0 + r * d, d, slot0 + r * P, P); r += 1; }
                    for (; r < r_c; ++r) stage(N1{}, Strided{}, Checked{}, pos0 + r * d, d, slot0 + r * P, P);
                    for (; r < n_rows; ++r) s_x[slot0 + r * P] = 0.0f;
                }
            }
            __syncthreads();
            static_assert(kWalkFeatures == 8, "two groups of four features");
            if (groups == 1) walk_tile<1>(s_x, P, cols, rows, seg_rows, ta, ca, t_min, t_full, c_more, w, b, cnt);
            else walk_tile<2>(s_x, P, cols, rows, seg_rows, ta, ca, t_min, t_full, c_more, w, b, cnt);
        }
    }
#pragma unroll
    for (int f = 0; f < kWalkFeatures; ++f) {
        const int v = __reduce_add_sync(0xffffffffu, cnt[f]);
        if ((tid & 31) == 0 && v) atomicAdd(&s_cnt[f], v);
    }
    __syncthreads();
    if (tid < nf) feat[(size_t)n * F + it.f0 + tid] = (float)s_cnt[tid] / (float)(last - first);   // Eq. 2
}

// Tiling of the dilated view for dilation d: the cheapest of the candidates under a simple cost model (staged
// samples, and thread slots of the walks including the ones that idle in a partly filled round of the block).
// Tiles either span whole rows (width = d) or 256-column multiples; runs are multiples of the window length;
// below 32 columns only run lengths that keep the lanes of a warp on different shared-memory banks.
void choose_walk(int d, int L, int& width, int& seg_rows, int& segs) {
    const int T = (L + d - 1) / d;
    const double c_stage = 17.0, c_walk = 21.0, c_fill = 16.0;
    double best = 1e300;
    width = 0;
    auto consider = [&](int w, int sr, int sg) {
        if ((int64_t)(sg * sr + 8) * w > kWalkSamples) return;
        const int tile_rows = sr * sg;
        double cost = 0.0;
        for (int ta = 0; ta < T; ta += tile_rows) {
            const int rows = std::min(tile_rows, T - ta), sgt = (rows + sr - 1) / sr;
            for (int ca = 0; ca < d; ca += w) {
                const int cols = std::min(w, d - ca);
                const double rounds = std::ceil((double)cols * sgt / kWalkThreads);
                cost += (double)(rows + 8) * cols * c_stage + rounds * kWalkThreads * (std::min(sr, rows) * c_walk + c_fill);
            }
        }
        if (cost < best) { best = cost; width = w; seg_rows = sr; segs = sg; }
    };
    for (int sr = kWalkLen; sr <= 7 * kWalkLen; sr += kWalkLen) {
        if (d < 32 && sr != 3 * kWalkLen && sr != 7 * kWalkLen) continue;
        const int max_segs = std::max(1, (T + sr - 1) / sr);
        for (int sg = 1; sg <= max_segs; sg = sg < 8 ? sg + 1 : sg * 2) consider(d, sr, sg);
        consider(d, sr, max_segs);
        if (kWalkSamples / d - 8 >= sr) consider(d, sr, std::min(max_segs, (kWalkSamples / d - 8) / sr));
        for (int w = kWalkThreads; w < d; w += kWalkThreads)
            for (int sg = 1; sg <= std::min(max_segs, 4); ++sg) consider(w, sr, sg);
    }
}

}  // namespace
}  // namespace fast
}  // namespace rocket
