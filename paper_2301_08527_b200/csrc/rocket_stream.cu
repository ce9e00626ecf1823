// Fused kernel of the large dilations: every warp streams its own tiles.
//
// With u = t d + r a dilated convolution is a dense filter down the columns of A[t][r] = x[t d + r].  A warp's tile is R rows
// (16, 12 or 8) x 64 columns of outputs of one kernel; a thread owns two neighbouring columns, R packed accumulators.  The
// kernel's channels come one after the other: the R + len - 1 input rows of a channel are ONE tiled bulk copy into the warp's
// own shared memory (two stages of 7 KB per warp), issued by one of its lanes as soon as the stage has been read for the last
// time, two (tile, channel) visits ahead, across tiles and units of work.  A warp waits on its own barriers only: no block
// barrier, no producer warp, no other warp's pace.
//
// Why: kernels of large dilation share no samples worth sharing, so a block-wide tile only couples its warps.  The earlier form
// (a producer warp, eight consumer warps behind a two-stage ring, 128 x 64 tiles; rocket_fast_fwd.cu) spent 16 of its 34 ms
// outside the multiplications - doing them twice cost 18 ms more - because a stage is free only when the slowest warp has read
// it, and 28 % (20 x 50,000) to 45 % (20 x 5,000) of the products lay outside a kernel's rows and columns.  Bytes: a visit
// brings R + len - 1 rows for R rows of outputs, 0.65 B per multiply-add, 55 B/clk/SM at the rate reached; bulk copies of
// this size deliver 75.  Heights of 16, 12 and 8 rows fit the output range to four rows.
//
// One copy for all rows of a tile: row s starts at position P + s d of the zero-margined row, and a bulk copy needs 16-byte
// aligned starts.  The rows exist in seven copies, copy j moved down by j floats, one after the other per channel row, so
// "next copy" is a stride like any other: for an odd dilation rows s = 4 y + i with i = 0..3 are a tensor dimension of stride
// pitch + d - 1 (d = 1 mod 4) or, counted backwards, pitch - d - 1 (d = 3 mod 4), and y one of stride 4 d; for d = 2 mod 4 rows
// come in pairs, for d = 0 mod 4 one by one.  Rows before the first and after the last y that holds samples are filled with
// zeros by the copy engine.
#include <algorithm>

#include "rocket_fast.h"
#include "rocket_fast_dev.cuh"
#include "rocket_fast_geom.h"

namespace rocket {
namespace fast {
namespace {

extern __shared__ __align__(128) unsigned char smem_raw[];

static_assert(kWStages == 2, "the producer runs less than a whole unit of one visit ahead");

// The channel loop either chooses the inner loop of the tile's shape for every channel, or exists once per shape as a whole (WHOLE).
// As a whole a channel costs less (soft transform of 32 x 20 x 50,000 33.1 -> 32.1 ms, backward 67.1 -> 65.6), but there is more
// code to fetch, which launches of a few dozen visits per warp do not make up for (10 x 6 x 1,251: 89 -> 97 us; even at 160
// visits per warp).  The hard modes, whose other code is small, lose by it at every size.
constexpr int kWWholeVisits = 300;

struct StreamArgs {
    FwdArgs f;
    const WUnit* units;
    int n_units;
    const void* maps;
    int examples, groups, groups_per_set;   // examples of an item; groups of examples of the pass; groups handed out together
};

// The inner loop: one channel of a warp tile, weights handed round from lane j (conv_channel with the weight already loaded).
template <int ELL, int R>
__device__ __forceinline__ void stream_conv(const float* __restrict__ st, const int (&off)[4], float mine, u64 (&acc)[kWRows]) {
    u64 wp[ELL];
#pragma unroll
    for (int j = 0; j < ELL; ++j) {
        const float w = __shfl_sync(kFull, mine, j);
        wp[j] = pack2(w, w);
    }
#pragma unroll
    for (int s = 0; s < R + ELL - 1; ++s) {
        const u64 x = *reinterpret_cast<const u64*>(st + off[s & 3] + (s >> 2) * (4 * kWarpCols));
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) fma2(acc[o], wp[j], x);
        }
    }
}
template <int ELL, int R>
__device__ __forceinline__ void stream_conv(const float* __restrict__ st, const int (&off)[4], float mine, h2 (&acc)[kWRows]) {
    const h2 mh = to_h2(mine, mine);
    h2 wp[ELL];
#pragma unroll
    for (int j = 0; j < ELL; ++j) wp[j] = __shfl_sync(kFull, mh, j);
#pragma unroll
    for (int s = 0; s < R + ELL - 1; ++s) {
        const float2 xf = *reinterpret_cast<const float2*>(st + off[s & 3] + (s >> 2) * (4 * kWarpCols));
        const h2 x = to_h2(xf.x, xf.y);
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) hfma2(acc[o], wp[j], x);
        }
    }
}

// What a lane carries from tile to tile of a unit.
struct Carry {
    int cnt;          // hard: outputs above zero
    float mn;         // hard, soft: min of -z
    u64 hsum;         // soft: sum of h, fixed point
    int idx;          // soft: lowest output index attaining the max
    long long db;     // backward: sum of gz, fixed point
};

// One channel of the second half of the backward: dw[j] += gz[o] x[o + j].
template <int ELL, int R>
__device__ __forceinline__ void stream_grad(const float* __restrict__ st, const int (&off)[4], const u64 (&gz)[kWRows], u64 (&dw)[ROCKET_MAX_LENGTH]) {
#pragma unroll
    for (int s = 0; s < R + ELL - 1; ++s) {
        const u64 x = *reinterpret_cast<const u64*>(st + off[s & 3] + (s >> 2) * (4 * kWarpCols));
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) fma2(dw[j], gz[o], x);
        }
    }
}

// Calls f(length, rows) as compile-time constants for shape = 3 * (length index) + (rows index).
template <typename F>
__device__ __forceinline__ void by_shape(int shape, F&& f) {
    using L7 = std::integral_constant<int, 7>;
    using L9 = std::integral_constant<int, 9>;
    using L11 = std::integral_constant<int, 11>;
    using R16 = std::integral_constant<int, 16>;
    using R12 = std::integral_constant<int, 12>;
    using R8 = std::integral_constant<int, 8>;
    switch (shape) {
        case 0: f(L7{}, R16{}); break;
        case 1: f(L7{}, R12{}); break;
        case 2: f(L7{}, R8{}); break;
        case 3: f(L9{}, R16{}); break;
        case 4: f(L9{}, R12{}); break;
        case 5: f(L9{}, R8{}); break;
        case 6: f(L11{}, R16{}); break;
        case 7: f(L11{}, R12{}); break;
        default: f(L11{}, R8{}); break;
    }
}

// The pooling works on the first R rows of the accumulators, four at a time from the eighth on (R is the same for the warp): one
// instance of it serves every shape, which keeps the code that the warps of an SM run at a time small.
template <typename F>
__device__ __forceinline__ void for_rows(int R, F&& row) {
#pragma unroll
    for (int o = 0; o < 8; ++o) row(o);
    if (R > 8) {
#pragma unroll
        for (int o = 8; o < 12; ++o) row(o);
        if (R > 12) {
#pragma unroll
            for (int o = 12; o < 16; ++o) row(o);
        }
    }
}

// Hard pooling: the count of set sign bits and the minimum of -z; outputs that do not exist count as +inf.
__device__ __forceinline__ void pool_hard_lane(const u64 (&acc)[kWRows], int R, bool interior, unsigned m0, unsigned m1, Carry& st) {
    const float inf = __int_as_float(0x7f800000);
    unsigned signs = 0;
    if (interior) {
        for_rows(R, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            signs = __funnelshift_l(__float_as_uint(a), signs, 1);
            signs = __funnelshift_l(__float_as_uint(b), signs, 1);
            st.mn = min3(st.mn, a, b);
        });
    } else {
        for_rows(R, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            a = (m0 & (1u << o)) ? a : inf;
            b = (m1 & (1u << o)) ? b : inf;
            signs = __funnelshift_l(__float_as_uint(a), signs, 1);
            signs = __funnelshift_l(__float_as_uint(b), signs, 1);
            st.mn = min3(st.mn, a, b);
        });
    }
    st.cnt += __popc(signs);
}

// Soft pooling of a tile into the lane's state (the sum as a fixed-point integer: exact and order-free from here on).
__device__ __forceinline__ void pool_soft_lane(const u64 (&acc)[kWRows], int R, float c1, float c0, bool interior, unsigned m0, unsigned m1,
                                               int base, int step, Carry& st) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f);
    u64 hs = pack2(0.0f, 0.0f);
    float mt = __int_as_float(0x7f800000);
    for_rows(R, [&](int o) {
        u64 t = c0p;
        fma2(t, acc[o], c1p);
        float ta, tb, a, b;
        unpack2(t, ta, tb);
        const u64 den = add2(pack2(ex2_approx(ta), ex2_approx(tb)), one);
        unpack2(den, ta, tb);
        float ha = rcp_approx(ta), hb = rcp_approx(tb);
        if (!interior) {
            if (!(m0 & (1u << o))) ha = 0.0f;
            if (!(m1 & (1u << o))) hb = 0.0f;
        }
        hs = add2(hs, pack2(ha, hb));
        unpack2(acc[o], a, b);
        mt = min3(mt, a, b);
    });
    float h0, h1;
    unpack2(hs, h0, h1);
    st.hsum += __float2ull_rn((h0 + h1) * kSoftFixedScale);
    if (mt <= st.mn && mt < __int_as_float(0x7f800000)) {
        int idx = INT_MAX;
        for_rows(R, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            if (a == mt) idx = min(idx, base + o * step);
            if (b == mt) idx = min(idx, base + 1 + o * step);
        });
        if (mt < st.mn || idx < st.idx) st.idx = idx;
        st.mn = mt;
    }
}

// Backward: the accumulators (-z) become gz in place; returns the thread's sum of them (see make_gz).
__device__ __forceinline__ float make_gz_lane(u64 (&acc)[kWRows], int R, float c1, float c0, float gPs, float gM, bool interior, unsigned m0,
                                              unsigned m1, int oA0, int oA1) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f), neg1 = pack2(-1.0f, -1.0f), gp = pack2(gPs, gPs);
    u64 sum = pack2(0.0f, 0.0f);
    for_rows(R, [&](int o) {
        u64 t = c0p;
        fma2(t, acc[o], c1p);
        float ta, tb;
        unpack2(t, ta, tb);
        const u64 den = add2(pack2(ex2_approx(ta), ex2_approx(tb)), one);
        unpack2(den, ta, tb);
        const u64 hh = pack2(rcp_approx(ta), rcp_approx(tb));
        u64 omh = one;
        fma2(omh, hh, neg1);                      // 1 - h
        u64 g = mul2(mul2(hh, omh), gp);
        float ga, gb;
        unpack2(g, ga, gb);
        if (!interior) {
            if (!(m0 & (1u << o))) ga = 0.0f;
            if (!(m1 & (1u << o))) gb = 0.0f;
        }
        if (o == oA0) ga += gM;
        if (o == oA1) gb += gM;
        g = pack2(ga, gb);
        acc[o] = g;
        sum = add2(sum, g);
    });
    float s0, s1;
    unpack2(sum, s0, s1);
    return s0 + s1;
}

__device__ __forceinline__ void publish_soft(unsigned long long* __restrict__ ws, int64_t pair, const Carry& st, int lane) {
    u64 hsum = st.hsum;
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) hsum += __shfl_xor_sync(kFull, hsum, sh);
    const int key = float_key(-st.mn), wkey = __reduce_max_sync(kFull, key);
    const int idx = __reduce_min_sync(kFull, key == wkey ? st.idx : INT_MAX);
    if (lane == 0) {
        atomicAdd(ws + 2 * pair, hsum);
        const unsigned long long k64 = ((unsigned long long)((unsigned)wkey ^ 0x80000000u) << 32) |
                                       (unsigned long long)(unsigned)(INT_MAX - idx);
        atomicMax(ws + 2 * pair + 1, k64);
    }
}

// The rest of a wait that did not succeed at once (out of line: the fast path is one test).
__device__ __noinline__ bool stream_wait_slow(uint32_t bar, uint32_t parity) { return mbar_wait(bar, parity); }

// Announces `bytes` on the barrier and starts the copy of one box, by one lane (lead != 0), without a branch.
__device__ __forceinline__ void stream_copy_box(int lead, uint32_t dst, const void* tmap, int x, int y, int w, uint32_t bar, uint32_t bytes) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.s32 p, %0, 0;\n\t"
        "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%6], %7;\n\t"
        "@p cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%1], [%2, {%3, 0, %4, %5}], [%6];\n\t}"
        ::"r"(lead), "r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(w), "r"(bar), "r"(bytes) : "memory");
}

template <int MODE, bool WHOLE = false>  // 0 = hard, 1 = soft, 2 = backward of soft, 3 = hard in half precision; WHOLE: see kWWholeVisits
__global__ void __launch_bounds__(kWThreads, 1) fast_stream(const __grid_constant__ StreamArgs a) {
    __shared__ unsigned long long s_bar[kWWarps][kWStages];
    const int lane = threadIdx.x & 31, warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
    const uint32_t raw = smem_u32(smem_raw);
    float* stages = reinterpret_cast<float*>(smem_raw + (((raw + 127u) & ~127u) - raw)) + warp * kWStages * kWStageFloats;
    const uint32_t stages0 = smem_u32(stages), bar0 = smem_u32(s_bar[warp]);
    if (lane == 0) {
        for (int i = 0; i < kWStages; ++i) mbar_init(bar0 + 8u * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();

    // An item of work is a unit for a group of examples.  Items run over the groups of a set (whose copies stay in L2) for
    // one unit, then over the units, then over the sets: the warps of a moment share a unit, its inner loop, weights and
    // tensor map.  The first item of a warp goes by its place, the others by a counter.  v, vn: the unit at work and the next
    // one, a word per lane (all zero past the last); drawn: the number of the item after that.
    const unsigned n_units = (unsigned)a.n_units, total = (unsigned)a.groups * n_units, warps = gridDim.x * kWWarps;
    unsigned* counter = a.f.plan.counters + 1;
    auto item = [&](unsigned g, int& n0) {             // unit of item g, and its first example
        const unsigned per_set = (unsigned)a.groups_per_set * n_units, set = g / per_set, rest = g - set * per_set;
        const unsigned first = set * (unsigned)a.groups_per_set, in_set = min((unsigned)a.groups_per_set, (unsigned)a.groups - first);
        const unsigned unit = rest / in_set;
        n0 = (int)(first + rest - unit * in_set) * a.examples;
        return unit;
    };
    auto load_unit = [&](unsigned g, int& n0) {
        n0 = 0;
        if (g >= total) return 0;
        return __ldg(reinterpret_cast<const int*>(a.units + item(g, n0)) + lane);
    };
    unsigned g = (unsigned)warp * gridDim.x + blockIdx.x, gn = 0, drawn = 0;
    if (g >= total) return;
    if (lane == 0) gn = warps + atomicAdd(counter, 1u);
    int n0, nn0;                                       // first example of v and of vn
    int v = load_unit(g, n0);
    if (lane == 0) drawn = warps + atomicAdd(counter, 1u);
    gn = __shfl_sync(kFull, gn, 0);
    int vn = load_unit(gn, nn0);

    // ---- producer side: issues the copy of one visit, two visits ahead of the multiplications, into the stage just read
    int pv = v, p_q = 0, p_visits = 0;                 // its unit's words; visit of the tile, visits per tile
    int p_tiles = 0, p_examples = 0;                   // tiles left of the example, examples left of the item
    int p_x = 0, p_y = 0, p_col = 0, p_rows = 0;       // box of the tile; lane q: copy row of channel q (of the q-th visit)
    uint32_t p_bytes = 0;
    const char* p_map = nullptr;
    auto pfield = [&](int i) { return __shfl_sync(kFull, pv, i); };
    auto p_tile = [&](int tile) {                      // the box of tile number `tile`
        const int ncol = pfield(18), band = tile / ncol, run = pfield(22);
        p_col = tile - band * ncol;
        p_x = pfield(20) + kWarpCols * p_col;
        p_y = pfield(21) + band * pfield(19);
        while (p_x >= run) { p_x -= run; ++p_y; }
    };
    auto aim = [&](int first) {                        // the unit in pv, from example `first` on; false: there is none
        const int m = pfield(7);
        if (m == 0) return false;
        p_visits = MODE == 2 ? 2 * m : m;              // the backward takes the channels twice
        p_q = 0;
        p_tiles = pfield(4);
        p_examples = min(a.examples, a.f.N - first);
        p_bytes = (uint32_t)pfield(27);
        const int q = MODE == 2 && lane >= m ? lane - m : lane;
        p_rows = (first * a.f.C + ((__shfl_sync(kFull, pv, 24 + ((q & 15) >> 2)) >> (8 * (q & 3))) & 0xff)) * kWCopies + pfield(23);
        p_tile(pfield(3));
        p_map = reinterpret_cast<const char*>(a.maps) + (size_t)pfield(1) * 128;
        return true;
    };
    auto advance = [&]() {                             // to the next tile; false when no work is left
        p_q = 0;
        if (--p_tiles > 0) {
            p_x += kWarpCols;
            if (++p_col == pfield(18)) p_tile(pfield(3) + pfield(4) - p_tiles);
            const int run = pfield(22);
            while (p_x >= run) { p_x -= run; ++p_y; }
            return true;
        }
        if (--p_examples > 0) {
            p_tiles = pfield(4);
            p_rows += a.f.C * kWCopies;
            p_tile(pfield(3));
            return true;
        }
        pv = vn;
        if (aim(nn0)) return true;
        p_visits = 0;                                  // asked again after every visit that is left
        p_tiles = p_examples = 1;
        return false;
    };
    auto issue = [&](uint32_t slot) {
        if (p_q == p_visits && !advance()) return;
        const int w = __shfl_sync(kFull, p_rows, p_q);
        stream_copy_box(lane == 0, stages0 + slot * (kWStageFloats * 4), p_map, p_x, p_y, w, bar0 + 8u * slot, p_bytes);
        ++p_q;
    };
    aim(n0);
    issue(0);
    issue(1);

    uint32_t st = 0;                                   // visits consumed: stage st & 1, parity st >> 1 & 1
    bool ok = true;
    auto wait = [&]() {
        const uint32_t bar = bar0 + 8u * (st & 1u), parity = (st >> 1) & 1u;
        return mbar_try(bar, parity) || stream_wait_slow(bar, parity);
    };
    const int weight_lane = 2 * min(lane, ROCKET_MAX_LENGTH - 1);
    int krec = __shfl_sync(kFull, v, 0);
    float w_first = __ldg(&a.f.plan.krec[krec].w2[0][0] + weight_lane), negb = __ldg(&a.f.plan.krec[krec].negb);
    while (g < total) {
        auto field = [&](int i) { return __shfl_sync(kFull, v, i); };
        const int t0 = field(2), tile0 = field(3), ntiles = field(4), shape = field(5), d = field(6), m = field(7), k = field(8);
        const int ncol = field(18), R = shape & 0xff, len = (shape >> 8) & 0xff, row_xor = (shape >> 16) & 3;
        const int index = 3 * ((len - 7) >> 1) + ((16 - R) >> 2);
        const float* __restrict__ wl = &a.f.plan.krec[krec].w2[0][0] + weight_lane;
        const int off[4] = {(0 ^ row_xor) * kWarpCols + 2 * lane, (1 ^ row_xor) * kWarpCols + 2 * lane,
                            (2 ^ row_xor) * kWarpCols + 2 * lane, (3 ^ row_xor) * kWarpCols + 2 * lane};
        const int examples = min(a.examples, a.f.N - n0), band0 = tile0 / ncol, col0 = tile0 - band0 * ncol;
        int next_krec = 0;
        float w_first_n = 0.0f, negb_n = 0.0f;
        Carry carry{0, __int_as_float(0x7f800000), 0ull, INT_MAX, 0ll};
        const double scale = MODE == 2 ? __ldg(a.f.scale + k) : 0.0;
        for (int e = 0; e < examples && ok; ++e) {
            const int64_t pair = (int64_t)(n0 + e) * a.f.K + k;
            float gP = 0.0f, gM = 0.0f;
            int tA = 0, cA = 0;
            if (MODE == 2) {
                gP = __ldg(a.f.dfeat + 2 * pair) * a.f.lambda / (float)field(16);
                gM = __ldg(a.f.dfeat + 2 * pair + 1);
                const int uA = __ldg(a.f.argmax + pair) - field(11);
                tA = uA / d;                           // floor division: uA >= -p may be negative
                cA = uA - tA * d;
                if (cA < 0) { cA += d; --tA; }
            }
            int col = col0, trow = t0 + band0 * R;
            for (int t = 0; t < ntiles; ++t) {
                const bool last = t + 1 == ntiles && e + 1 == examples;      // of the item
                const int c0 = col * kWarpCols, c = c0 + 2 * lane;
                const bool interior = tile_interior(trow, c0, field(28), d, field(9), field(10));
                unsigned m0 = 0, m1 = 0;               // rows of the lane's two columns that are outputs
                if (!interior) {
                    const int tl = field(12), rl = field(13), th = field(14), rh = field(15);
                    int lo, hi;
                    valid_rows_tc(trow, c, tl, rl, th, rh, R, c < d, lo, hi);
                    m0 = row_mask(lo, hi);
                    valid_rows_tc(trow, c + 1, tl, rl, th, rh, R, c + 1 < d, lo, hi);
                    m1 = row_mask(lo, hi);
                }
                u64 acc[kWRows];
                [[maybe_unused]] h2 acch[kWRows];
                if constexpr (MODE == 3) {
                    init_acc_h(acch, negb);
                } else if (MODE == 0 || interior) {
                    const u64 start = pack2(negb, negb);
#pragma unroll
                    for (int o = 0; o < kWRows; ++o) acc[o] = start;
                } else {                               // +inf where there is no output
                    const float inf = __int_as_float(0x7f800000);
#pragma unroll
                    for (int o = 0; o < kWRows; ++o) acc[o] = pack2((m0 & (1u << o)) ? negb : inf, (m1 & (1u << o)) ? negb : inf);
                }
                float mine = w_first;
                const float* __restrict__ wn = wl;
                auto channel = [&](int q, auto&& conv) {
                    if (q + 1 < m) wn += kPairRow;
                    const float mine_next = __ldg(wn);
                    if (!(ok = wait())) return false;
                    const uint32_t slot = st & 1u;
                    conv(stages + slot * kWStageFloats);
                    mine = mine_next;
                    __syncwarp();                      // the stage has been read by every lane
                    ++st;
                    if (MODE == 2 || !last || q + 1 < m) issue(slot);
                    return true;
                };
                if constexpr (WHOLE) {
                    by_shape(index, [&](auto len_tag, auto r_tag) {
                        for (int q = 0; q < m; ++q)
                            if (!channel(q, [&](const float* stage) { stream_conv<decltype(len_tag)::value, decltype(r_tag)::value>(stage, off, mine, acc); })) break;
                    });
                } else {
                    for (int q = 0; q < m; ++q) {
                        if (!channel(q, [&](const float* stage) {
                                by_shape(index, [&](auto len_tag, auto r_tag) {
                                    if constexpr (MODE == 3) stream_conv<decltype(len_tag)::value, decltype(r_tag)::value>(stage, off, mine, acch);
                                    else stream_conv<decltype(len_tag)::value, decltype(r_tag)::value>(stage, off, mine, acc);
                                });
                            })) break;
                    }
                }
                if (!ok) break;
                if constexpr (MODE == 3) widen_acc(acch, acc);
                if constexpr (MODE == 2) {
                    const bool hit = tA >= trow && tA < trow + R;
                    const float dbs = make_gz_lane(acc, R, a.f.c1, a.f.c0, gP, gM, interior, m0, m1, hit && c < d && c == cA ? tA - trow : -1,
                                                   hit && c + 1 < d && c + 1 == cA ? tA - trow : -1);
                    carry.db += __double2ll_rn((double)dbs * scale);
                    long long* dst = a.f.accfix + field(17);
                    for (int q = 0; q < m; ++q, dst += len) {
                        if (!(ok = wait())) break;
                        const uint32_t slot = st & 1u;
                        u64 dw[ROCKET_MAX_LENGTH];
#pragma unroll
                        for (int j = 0; j < ROCKET_MAX_LENGTH; ++j) dw[j] = 0ull;
                        by_shape(index, [&](auto len_tag, auto r_tag) {
                            stream_grad<decltype(len_tag)::value, decltype(r_tag)::value>(stages + slot * kWStageFloats, off, acc, dw);
                        });
                        __syncwarp();
                        ++st;
                        if (!last || q + 1 < m) issue(slot);
                        reduce_publish_dw<ROCKET_MAX_LENGTH>(dw, dst, scale, lane, len);
                    }
                    if (!ok) break;
                } else if constexpr (MODE == 1) {
                    pool_soft_lane(acc, R, a.f.c1, a.f.c0, interior, m0, m1, trow * d + c + field(11), d, carry);
                } else {
                    pool_hard_lane(acc, R, interior, m0, m1, carry);
                }
                if (++col == ncol) { col = 0; trow += R; }
            }
            if (!ok) break;
            if (e == 0) {                              // what the next unit needs first is on its way
                next_krec = __shfl_sync(kFull, vn, 0);
                w_first_n = __ldg(&a.f.plan.krec[next_krec].w2[0][0] + weight_lane);
                negb_n = __ldg(&a.f.plan.krec[next_krec].negb);
            }
            if (e + 1 < examples && MODE != 2) {
                if (MODE == 1) publish_soft(a.f.ws, pair, carry, lane);
                else publish(a.f.feat_i, pair, carry.cnt, carry.mn, lane);
                carry = Carry{0, __int_as_float(0x7f800000), 0ull, INT_MAX, 0ll};
            }
        }
        if (!ok) break;
        // the next item takes over, and the visit that this one's last still owes is issued
        const int64_t last_pair = (int64_t)(n0 + examples - 1) * a.f.K + k;
        v = vn;
        g = gn;
        n0 = nn0;
        krec = next_krec;
        w_first = w_first_n;
        negb = negb_n;
        gn = __shfl_sync(kFull, drawn, 0);
        vn = load_unit(gn, nn0);
        if (lane == 0) drawn = warps + atomicAdd(counter, 1u);
        issue((st - 1u) & 1u);
        if (MODE == 1) {
            publish_soft(a.f.ws, last_pair, carry, lane);
        } else if (MODE == 2) {
            long long db = carry.db;
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) db += __shfl_xor_sync(kFull, db, sh);
            if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(a.f.accfix + a.f.n_weights + k), (unsigned long long)db);
        } else {
            publish(a.f.feat_i, last_pair, carry.cnt, carry.mn, lane);
        }
    }
    if (!ok) {
        // a wait gave up: the results are incomplete, and nothing of this warp may be in flight when the block ends
        if (lane == 0) atomicExch(a.f.plan.error_flag, 1);
        for (int i = 0; i < kWStages; ++i, ++st) stream_wait_slow(bar0 + 8u * (st & 1u), (st >> 1) & 1u);
    }
    // Begun early, this kernel may end before the S kernel does.  Its last block waits for the S kernel here (it has a warp with work),
    // so that what follows in the stream, or behind this kernel's node of a captured graph, follows the S kernel too.  The last alone:
    // blocks that wait keep their SMs from the blocks still to come (10 x 6 x 1,251, both training passes: 194 us, 214 with a wait
    // in every block).
    if (blockIdx.x == gridDim.x - 1) dependency_wait();
}

size_t stream_smem_bytes() { return (size_t)kWWarps * kWStages * kWStageFloats * sizeof(float) + 128; }

}  // namespace

cudaError_t set_stream_attributes() {
    const int bytes = (int)stream_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(fast_stream<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fast_stream<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fast_stream<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fast_stream<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fast_stream<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fast_stream<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e;
}

void launch_stream(const FwdArgs& f, int mode, int sms, int64_t l2_bytes, bool after_s, cudaStream_t stream) {
    StreamArgs a;
    a.f = f;
    a.units = f.plan.wunits;
    a.n_units = f.plan.n_wunits;
    a.maps = f.plan.wmaps;
    const StreamItems it = stream_items(f.N, f.C, f.L, a.n_units, f.plan.w_visits, mode, sms, l2_bytes);
    a.examples = it.examples;
    a.groups = it.groups;
    a.groups_per_set = it.groups_per_set;
    const unsigned long long items = (unsigned long long)a.groups * (unsigned long long)a.n_units;
    const unsigned grid = (unsigned)std::min<unsigned long long>((items + kWWarps - 1) / kWWarps, (unsigned long long)sms);
    const size_t bytes = stream_smem_bytes();
    const bool whole = f.plan.w_visits * f.N >= (double)kWWholeVisits * sms * kWWarps;
    // Behind the S kernel this one may begin as SMs run out of S tiles: every block of the S kernel has by then seen the kernels before
    // it complete, and those wrote all that this one reads.
    auto launch = [&](auto kernel) {
        if (after_s) launch_dependent(kernel, grid, kWThreads, bytes, stream, a);
        else kernel<<<grid, kWThreads, bytes, stream>>>(a);
    };
    if (mode == 1 && whole) launch(fast_stream<1, true>);
    else if (mode == 1) launch(fast_stream<1>);
    else if (mode == 2 && whole) launch(fast_stream<2, true>);
    else if (mode == 2) launch(fast_stream<2>);
    else if (mode == 3) launch(fast_stream<3>);
    else launch(fast_stream<0>);
    count_launch();
}

}  // namespace fast
}  // namespace rocket
