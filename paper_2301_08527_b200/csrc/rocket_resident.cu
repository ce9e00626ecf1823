// Fused kernel of short series: whole examples in shared memory, every dilation in one launch.
//
// With u = t d + r a dilated convolution is a dense filter down the columns of A[t][r] = x[t d + r].  A block brings one or more whole
// examples (all channels, zeros between the rows as far as there is room) into shared memory and its warps take (kernel, example) pairs one by
// one, or parts of them where there are few; the parts of a pair meet in shared memory, so that features are written once and finally: no
// initialising and finalising kernels, no staging copies, no workspace.  A pair's outputs are cut into bands of two heights, in the
// backward of one (see resident_high), from its own first output on; a warp tile is 64 neighbouring columns of the bands strung together, a lane
// owns columns lane and lane + 32 as packed pairs.
//
// Why: the other kernels copy a tile per dilation (or per kernel) to use it for a handful of kernels, in bands of at least 8 rows that
// short series do not fill.  24 x 32 x 1,751 with 2,000 kernels spent three quarters of its 477 us on copies and draws of tiles that 4 to
// 250 kernels shared; here an example is copied once for all of them.
//
// Bound: issue slots.  A row of a tile is two loads, two address steps and 7 to 11 packed multiply-adds (the dilation is no constant, so
// that addresses are no immediate offsets); what else counts is code, of which the warps of an SM should use as little as possible at a
// time: hence zeros beside the rows in place of tests, and kernels ordered by length and not by work (24 x 32 x 1,751 with 2,000 kernels 222 and
// 548 us, 100 x 20 x 1,400 with 4,000 1,339 and 1,577).  Measured (us, before and now): 24 x 32 x 1,751 with 2,000 kernels 476 and 222, 16 x 1 x 512
// with 1,000 36 and 18.5, 100 x 20 x 600 with 4,000 1,283 and 715, soft 1,166 and 444 (2,000
// kernels), backward of 24 x 9 x 700 with 2,000 374 and 229.
#include <algorithm>

#include "rocket_fast.h"
#include "rocket_fast_dev.cuh"
#include "rocket_fast_geom.h"

namespace rocket {
namespace fast {
namespace {

extern __shared__ __align__(128) unsigned char smem_raw[];

static_assert(resident_high(2) + ROCKET_MAX_LENGTH - 1 <= 31, "the row masks hold the input rows of a tile");

__device__ __forceinline__ void copy4(uint32_t dst, const void* src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void copy16(uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }

// *p in shared memory, or zero without touching it.
__device__ __forceinline__ float shared_if(uint32_t p, unsigned ok) {
    float v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@q ld.shared.f32 %0, [%1];\n\t}" : "=f"(v) : "r"(p), "r"(ok));
    return v;
}

// The lane's two columns of a tile in one channel: where their first rows lie (bytes from the start of shared memory), how far it is
// from row to row, and, unless all of them are samples, which input rows are.
struct Columns { unsigned a, b, step, ma, mb; };

template <int ROWS, bool INSIDE, typename F>
__device__ __forceinline__ void for_inputs(const Columns& at, F&& row) {
    const char* pa = reinterpret_cast<const char*>(smem_raw) + at.a;
    const char* pb = reinterpret_cast<const char*>(smem_raw) + at.b;
    uint32_t qa = smem_u32(pa), qb = smem_u32(pb);
#pragma unroll
    for (int s = 0; s < ROWS; ++s) {
        float xa, xb;
        if (INSIDE) {
            xa = *reinterpret_cast<const float*>(pa);
            xb = *reinterpret_cast<const float*>(pb);
            pa += at.step;
            pb += at.step;
        } else {
            xa = shared_if(qa, at.ma & (1u << s));
            xb = shared_if(qb, at.mb & (1u << s));
            qa += at.step;
            qb += at.step;
        }
        row(s, xa, xb);
    }
}

// Where the items of a pair that is divided meet: count and max key (hard), sum and (max key, INT_MAX - index) (soft), items still to come.
struct Merge { u64 sum; int cnt, key; u64 best; int left, pad; };
static_assert(sizeof(Merge) == 4 * kRMergeFloats, "room for them is counted in floats");

// What a lane keeps of a pair from tile to tile.
struct Pair {
    int cnt;          // hard: outputs above zero
    float mn;         // hard, soft: min of -z
    u64 hsum;         // soft: sum of h, fixed point
    int idx;          // soft: lowest output index attaining the max
    long long db;     // backward: sum of gz, fixed point
};

// What depends on the heights of the bands.
template <int HIGH, int LOW>
struct Bands {
static constexpr int kHigh = HIGH, kLow = LOW;

template <int ELL, int R, bool INSIDE>
static __device__ __forceinline__ void resident_conv(const Columns& at, float mine, u64 (&acc)[kHigh]) {
    u64 wp[ELL];
#pragma unroll
    for (int j = 0; j < ELL; ++j) {
        const float w = __shfl_sync(kFull, mine, j);
        wp[j] = pack2(w, w);
    }
    for_inputs<R + ELL - 1, INSIDE>(at, [&](int s, float xa, float xb) {
        const u64 x = pack2(xa, xb);
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) fma2(acc[o], wp[j], x);
        }
    });
}
template <int ELL, int R, bool INSIDE>
static __device__ __forceinline__ void resident_conv(const Columns& at, float mine, h2 (&acc)[kHigh]) {
    const h2 mh = to_h2(mine, mine);
    h2 wp[ELL];
#pragma unroll
    for (int j = 0; j < ELL; ++j) wp[j] = __shfl_sync(kFull, mh, j);
    for_inputs<R + ELL - 1, INSIDE>(at, [&](int s, float xa, float xb) {
        const h2 x = to_h2(xa, xb);
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) hfma2(acc[o], wp[j], x);
        }
    });
}
// One channel of the second half of the backward: dw[j] += gz[o] x[o + j].
template <int ELL, int R, bool INSIDE>
static __device__ __forceinline__ void resident_grad(const Columns& at, const u64 (&gz)[kHigh], u64 (&dw)[ROCKET_MAX_LENGTH]) {
    for_inputs<R + ELL - 1, INSIDE>(at, [&](int s, float xa, float xb) {
        const u64 x = pack2(xa, xb);
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const int o = s - j;
            if (o >= 0 && o < R) fma2(dw[j], gz[o], x);
        }
    });
}

// Calls f(length, rows, inside) as compile-time constants.
template <typename F>
static __device__ __forceinline__ void by_form(int len, bool high, bool inside, F&& f) {
    auto rows = [&](auto len_tag) {
        using High = std::integral_constant<int, kHigh>;
        using Low = std::integral_constant<int, kLow>;
        if (high) inside ? f(len_tag, High{}, std::true_type{}) : f(len_tag, High{}, std::false_type{});
        else inside ? f(len_tag, Low{}, std::true_type{}) : f(len_tag, Low{}, std::false_type{});
    };
    if (len == 7) rows(std::integral_constant<int, 7>{});
    else if (len == 9) rows(std::integral_constant<int, 9>{});
    else rows(std::integral_constant<int, 11>{});
}

// The first kLow or all kHigh rows of a tile (the same for the warp).
template <typename F>
static __device__ __forceinline__ void for_rows(bool high, F&& row) {
#pragma unroll
    for (int o = 0; o < kLow; ++o) row(o);
    if (high) {
#pragma unroll
        for (int o = kLow; o < kHigh; ++o) row(o);
    }
}

static __device__ __forceinline__ void pool_hard_rows(const u64 (&acc)[kHigh], bool high, bool all, unsigned m0, unsigned m1, Pair& st) {
    const float inf = __int_as_float(0x7f800000);
    unsigned s0 = 0, s1 = 0;
    if (all) {
        for_rows(high, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            s0 = __funnelshift_l(__float_as_uint(a), s0, 1);
            s1 = __funnelshift_l(__float_as_uint(b), s1, 1);
            st.mn = min3(st.mn, a, b);
        });
    } else {
        for_rows(high, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            a = (m0 & (1u << o)) ? a : inf;
            b = (m1 & (1u << o)) ? b : inf;
            s0 = __funnelshift_l(__float_as_uint(a), s0, 1);
            s1 = __funnelshift_l(__float_as_uint(b), s1, 1);
            st.mn = min3(st.mn, a, b);
        });
    }
    st.cnt += __popc(s0) + __popc(s1);
}

static __device__ __forceinline__ void pool_soft_rows(const u64 (&acc)[kHigh], bool high, float c1, float c0, bool all, unsigned m0, unsigned m1,
                                               int base0, int base1, int step, Pair& st) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f);
    u64 hs = pack2(0.0f, 0.0f);
    float mt = __int_as_float(0x7f800000);
    for_rows(high, [&](int o) {
        u64 t = c0p;
        fma2(t, acc[o], c1p);
        float ta, tb, a, b;
        unpack2(t, ta, tb);
        const u64 den = add2(pack2(ex2_approx(ta), ex2_approx(tb)), one);
        unpack2(den, ta, tb);
        float ha = rcp_approx(ta), hb = rcp_approx(tb);
        if (!all) {
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
        for_rows(high, [&](int o) {
            float a, b;
            unpack2(acc[o], a, b);
            if (a == mt) idx = min(idx, base0 + o * step);
            if (b == mt) idx = min(idx, base1 + o * step);
        });
        if (mt < st.mn || idx < st.idx) st.idx = idx;
        st.mn = mt;
    }
}

// Backward: the accumulators (-z) become gz in place (see make_gz); returns the thread's sum of them.
static __device__ __forceinline__ float make_gz_rows(u64 (&acc)[kHigh], bool high, float c1, float c0, float gPs, float gM, bool all, unsigned m0,
                                              unsigned m1, int oA0, int oA1) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f), neg1 = pack2(-1.0f, -1.0f), gp = pack2(gPs, gPs);
    u64 sum = pack2(0.0f, 0.0f);
    for_rows(high, [&](int o) {
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
        if (!all) {
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
};

template <int MODE, int BANDS>  // 0 = hard, 1 = soft, 2 = backward of soft, 3 = hard in half precision; BANDS: their heights
__global__ void __launch_bounds__(32 * resident_warps(MODE, BANDS), 1) fast_resident(const __grid_constant__ ResidentArgs a) {
    using B = Bands<resident_high(BANDS), resident_low(BANDS)>;
    constexpr bool kOneHeight = B::kHigh == B::kLow;
    constexpr int kWarps = resident_warps(MODE, BANDS), kHigh = B::kHigh, kLow = B::kLow;
    __shared__ int s_next;
    float* xs = reinterpret_cast<float*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned tasks = (unsigned)a.groups * (unsigned)a.parts;
    const int weight_lane = 2 * min(lane, ROCKET_MAX_LENGTH - 1);
    Merge* merge = reinterpret_cast<Merge*>(xs + a.front + a.examples * a.C * a.pitch);
    // zeros in front of the first channel row and behind every one, as far as the next; the samples never reach them
    for (int i = tid; i < a.front; i += 32 * kWarps) xs[i] = 0.0f;
    for (int row = warp; row < a.examples * a.C; row += kWarps)
        for (int i = a.L + lane; i < a.pitch; i += 32) xs[a.front + row * a.pitch + i] = 0.0f;
    for (unsigned task = blockIdx.x; task < tasks; task += gridDim.x) {
        const int group = (int)(task / (unsigned)a.parts), part = (int)(task - (unsigned)group * (unsigned)a.parts);
        const int n0 = group * a.examples, ne = min(a.examples, a.N - n0);
        __syncthreads();                               // the examples of the task before have been read
        if (tid == 0) s_next = 0;
        if (MODE != 2 && a.split_bits > 0)
            for (int i = tid; i < (a.n_units / a.parts + 1) * ne; i += 32 * kWarps) merge[i] = Merge{0ull, 0, INT_MIN, 0ull, 1 << a.split_bits, 0};
        for (int row = warp; row < ne * a.C; row += kWarps) {
            float* dst = xs + a.front + row * a.pitch;
            const size_t first = ((size_t)n0 * a.C + row) * a.L;
            if (a.X8) {                                // L and the base are multiples of four
                const float mu = a.norm.mean[row % a.C], is = a.norm.inv_std[row % a.C];
                const uchar4* __restrict__ src = reinterpret_cast<const uchar4*>(a.X8 + first);
                for (int i = lane; i < a.L / 4; i += 32) {
                    const uchar4 u = __ldg(src + i);
                    reinterpret_cast<float4*>(dst)[i] = make_float4(((float)u.x - mu) * is, ((float)u.y - mu) * is, ((float)u.z - mu) * is, ((float)u.w - mu) * is);
                }
            } else if (a.aligned) {                    // every row starts at a 16-byte boundary
                for (int i = lane; i < a.L / 4; i += 32) copy16(smem_u32(dst + 4 * i), a.X + first + 4 * i);
            } else {
#pragma unroll 4
                for (int i = lane; i < a.L; i += 32) copy4(smem_u32(dst + i), a.X + first + i);
            }
        }
        // Items: every parts-th kernel, for a few of the examples.  v, v1: the units of the item at work and of the next one, a word per
        // lane (all zero past the last); the number of the one after that is drawn, and its unit on its way, while an item is at work.
        const int n_kernels = (a.n_units - part + a.parts - 1) / a.parts, runs = (ne + a.run - 1) / a.run, n_items = (n_kernels * runs) << a.split_bits;
        auto draw = [&]() {
            int i = 0;
            if (lane == 0) i = atomicAdd(&s_next, 1);
            return __shfl_sync(kFull, i, 0);
        };
        auto load_unit = [&](int i, int& e) {
            e = 0;
            if (i >= n_items) return 0;
            i >>= a.split_bits;
            const int q = runs == 1 ? i : i / runs;
            e = (i - q * runs) * a.run;
            return __ldg(reinterpret_cast<const int*>(a.units + part + q * a.parts) + lane);
        };
        auto first_weight = [&](int unit) { return __ldg(&a.krec[__shfl_sync(kFull, unit, 0)].w2[0][0] + weight_lane); };
        auto bias_of = [&](int unit) { return __ldg(&a.krec[__shfl_sync(kFull, unit, 0)].negb); };
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        int e0, e1, e2;
        int i = draw(), i1 = draw();
        int v = load_unit(i, e0), v1 = load_unit(i1, e1);
        float w_first = first_weight(v), negb = bias_of(v);
        while (i < n_items) {
            const int i2 = draw(), v2 = load_unit(i2, e2);
            const float w_first_n = first_weight(v1), negb_n = bias_of(v1);   // what the next item needs first
            auto field = [&](int f) { return __shfl_sync(kFull, v, f); };
            const int krec = field(0), k = field(1), len = field(2), d = field(3), m = field(4), nout = field(5), p = field(6);
            const float* __restrict__ wl = &a.krec[krec].w2[0][0] + weight_lane;
            const int nq = field(9), nr = field(10), pq = field(11), pr = field(12), lq = field(13), lr = field(14);
            const float inv_d = __int_as_float(field(15));
            const int high_bands = kOneHeight ? (nq + (nr > 0) + kHigh - 1) / kHigh : field(7), low_bands = kOneHeight ? 0 : field(8);
            const unsigned row_bytes = 4u * (unsigned)a.pitch;
            const int e_end = min(ne, e0 + a.run);
            const double scale = MODE == 2 ? __ldg(a.scale + k) : 0.0;
            // the lane's columns of a tile: column of A, first row, the first row's output index, output rows there are, input rows there are
            int col[2], row0[2], i0[2], out[2];
            unsigned in[2], m0 = 0, m1 = 0;
            bool inside = false, all = false, known = false;
            const bool one_tile = high_bands == 0 ? low_bands * d <= kWarpCols : low_bands == 0 && high_bands * d <= kWarpCols;
            for (int e = e0; e < e_end; ++e) {
                const int64_t pair = (int64_t)(n0 + e) * a.K + k;
                const unsigned plane0 = 4u * ((unsigned)a.front + (unsigned)(e * a.C) * (unsigned)a.pitch);
                Pair st{0, __int_as_float(0x7f800000), 0ull, INT_MAX, 0ll};
                float gP = 0.0f, gM = 0.0f;
                int tA = 0, rA = 0;                    // the argmax as a row and a column counted from the first output
                const int others = (1 << a.split_bits) - 1;
                int tile = -i;                         // the item's are those whose number, so shifted, is a multiple of the items of a pair
                if (MODE == 2) {
                    gP = __ldg(a.dfeat + 2 * pair) * a.lambda / (float)nout;
                    gM = __ldg(a.dfeat + 2 * pair + 1);
                    const int at = __ldg(a.argmax_in + pair);
                    tA = at / d;
                    rA = at - tA * d;
                }
                for (int half = 0; half < (kOneHeight ? 1 : 2); ++half) {
                    const bool high = half == 0;
                    const int R = high ? kHigh : kLow, ncols = (high ? high_bands : low_bands) * d;
                    for (int c0 = 0; c0 < ncols; c0 += kWarpCols) {
                        if ((tile++ & others) != 0) continue;
                        if (!known) {
                            const int row_base = high ? 0 : kHigh * high_bands, rows = R + len - 1;
                            inside = true;
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const int c = c0 + lane + 32 * h;
                                const ResidentColumn at = resident_column(min(c, ncols - 1), row_base, R, len, d, inv_d, nq, nr, pq, pr, lq, lr);
                                row0[h] = at.row;
                                col[h] = at.r;
                                i0[h] = at.i0;
                                out[h] = c < ncols ? at.out : 0;
                                in[h] = row_mask(at.in_lo, at.in_hi);
                                inside = inside && at.in_lo == 0 && at.in_hi == rows;
                            }
                            inside = __all_sync(kFull, inside);
                            all = __all_sync(kFull, out[0] == R && out[1] == R);
                            m0 = row_mask(0, out[0]);
                            m1 = row_mask(0, out[1]);
                            if (!__any_sync(kFull, (out[0] | out[1]) != 0)) continue;
                            known = one_tile;
                        }
                        u64 acc[kHigh];
                        [[maybe_unused]] h2 acch[kHigh];
                        if constexpr (MODE == 3) {
                            init_acc_h(acch, negb);
                        } else if (MODE == 0 || all) {
                            const u64 start = pack2(negb, negb);
#pragma unroll
                            for (int o = 0; o < kHigh; ++o) acc[o] = start;
                        } else {                       // +inf where there is no output
                            const float inf = __int_as_float(0x7f800000);
#pragma unroll
                            for (int o = 0; o < kHigh; ++o) acc[o] = pack2((m0 & (1u << o)) ? negb : inf, (m1 & (1u << o)) ? negb : inf);
                        }
                        auto columns = [&](int q) {
                            const unsigned ch = (unsigned)field(16 + (q >> 2)) >> (8 * (q & 3)) & 0xffu, plane = plane0 + ch * row_bytes;
                            return Columns{plane + 4u * (unsigned)(i0[0] - p), plane + 4u * (unsigned)(i0[1] - p), 4u * (unsigned)d, in[0], in[1]};
                        };
                        float mine = w_first;
                        const float* __restrict__ wn = wl;
                        for (int q = 0; q < m; ++q) {
                            if (q + 1 < m) wn += kPairRow;
                            const float mine_next = __ldg(wn);
                            const Columns at = columns(q);
                            B::by_form(len, high, MODE == 2 || inside, [&](auto len_tag, auto r_tag, auto inside_tag) {
                                if constexpr (MODE == 3) B::template resident_conv<decltype(len_tag)::value, decltype(r_tag)::value, decltype(inside_tag)::value>(at, mine, acch);
                                else B::template resident_conv<decltype(len_tag)::value, decltype(r_tag)::value, decltype(inside_tag)::value>(at, mine, acc);
                            });
                            mine = mine_next;
                        }
                        if constexpr (MODE == 3) widen_acc(acch, acc);
                        if constexpr (MODE == 2) {
                            const int oA0 = col[0] == rA && tA >= row0[0] && tA < row0[0] + out[0] ? tA - row0[0] : -1;
                            const int oA1 = col[1] == rA && tA >= row0[1] && tA < row0[1] + out[1] ? tA - row0[1] : -1;
                            const float dbs = B::make_gz_rows(acc, high, a.c1, a.c0, gP, gM, all, m0, m1, oA0, oA1);
                            st.db += __double2ll_rn((double)dbs * scale);
                            long long* dst = a.accfix + field(19);
                            for (int q = 0; q < m; ++q, dst += len) {
                                u64 dw[ROCKET_MAX_LENGTH];
#pragma unroll
                                for (int j = 0; j < ROCKET_MAX_LENGTH; ++j) dw[j] = 0ull;
                                const Columns at = columns(q);
                                B::by_form(len, high, MODE == 2 || inside, [&](auto len_tag, auto r_tag, auto inside_tag) {
                                    B::template resident_grad<decltype(len_tag)::value, decltype(r_tag)::value, decltype(inside_tag)::value>(at, acc, dw);
                                });
                                reduce_publish_dw<ROCKET_MAX_LENGTH>(dw, dst, scale, lane, len);
                            }
                        } else if constexpr (MODE == 1) {
                            B::pool_soft_rows(acc, high, a.c1, a.c0, all, m0, m1, i0[0], i0[1], d, st);
                        } else {
                            B::pool_hard_rows(acc, high, all, m0, m1, st);
                        }
                    }
                }
                if constexpr (MODE == 2) {
                    long long db = st.db;
#pragma unroll
                    for (int sh = 16; sh > 0; sh >>= 1) db += __shfl_xor_sync(kFull, db, sh);
                    if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(a.accfix + a.n_weights + k), (unsigned long long)db);
                } else if constexpr (MODE == 1) {
                    u64 hsum = st.hsum;
#pragma unroll
                    for (int sh = 16; sh > 0; sh >>= 1) hsum += __shfl_xor_sync(kFull, hsum, sh);
                    const int key = float_key(-st.mn);
                    int wkey = __reduce_max_sync(kFull, key), idx = __reduce_min_sync(kFull, key == wkey ? st.idx : INT_MAX);
                    if (lane == 0) {
                        bool last = true;
                        if (a.split_bits > 0) {
                            Merge& at = merge[i >> a.split_bits];
                            atomicAdd(&at.sum, hsum);
                            atomicMax(&at.best, (u64)((unsigned)wkey ^ 0x80000000u) << 32 | (unsigned)(INT_MAX - idx));
                            __threadfence_block();
                            last = atomicSub(&at.left, 1) == 1;
                            __threadfence_block();
                            const u64 best = *(volatile u64*)&at.best;
                            hsum = *(volatile u64*)&at.sum;
                            wkey = (int)((unsigned)(best >> 32) ^ 0x80000000u);
                            idx = INT_MAX - (int)(unsigned)best;
                        }
                        if (last) {
                            a.feat[2 * pair] = (float)((double)hsum / (double)kSoftFixedScale / (double)nout);   // Eq. 4
                            a.feat[2 * pair + 1] = key_float(wkey);
                            if (a.argmax) a.argmax[pair] = idx;
                        }
                    }
                } else {
                    int cnt = __reduce_add_sync(kFull, st.cnt), key = __reduce_max_sync(kFull, float_key(-st.mn));
                    if (lane == 0) {
                        bool last = true;
                        if (a.split_bits > 0) {
                            Merge& at = merge[i >> a.split_bits];
                            atomicAdd(&at.cnt, cnt);
                            atomicMax(&at.key, key);
                            __threadfence_block();
                            last = atomicSub(&at.left, 1) == 1;
                            __threadfence_block();
                            cnt = *(volatile int*)&at.cnt;
                            key = *(volatile int*)&at.key;
                        }
                        if (last) {
                            a.feat[2 * pair] = (float)cnt / (float)nout;   // Eq. 2
                            a.feat[2 * pair + 1] = key_float(key);
                        }
                    }
                }
            }
            v = v1;
            v1 = v2;
            i = i1;
            i1 = i2;
            e0 = e1;
            e1 = e2;
            w_first = w_first_n;
            negb = negb_n;
        }
    }
}

}  // namespace

static cudaError_t allow_smem(std::initializer_list<void (*)(ResidentArgs)> kernels) {
    cudaError_t e = cudaSuccess;
    for (auto kernel : kernels)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRMostFloats * (int)sizeof(float));
    return e;
}
cudaError_t set_resident_attributes(int bands, bool backward) {
    if (backward) return allow_smem({bands == 3 ? fast_resident<2, 3> : bands == 4 ? fast_resident<2, 4> : bands == 5 ? fast_resident<2, 5> : fast_resident<2, 6>});
    return bands == 0   ? allow_smem({fast_resident<0, 0>, fast_resident<1, 0>, fast_resident<3, 0>})
           : bands == 1 ? allow_smem({fast_resident<0, 1>, fast_resident<1, 1>, fast_resident<3, 1>})
                        : allow_smem({fast_resident<0, 2>, fast_resident<1, 2>, fast_resident<3, 2>});
}

void launch_resident(ResidentArgs& a, const PlanHost& plan, int mode, int sms, cudaStream_t stream) {
    const ResidentSplit s = resident_split(plan, a.N, a.C, sms, mode);
    a.examples = s.examples;
    a.groups = s.groups;
    a.parts = s.parts;
    a.run = s.run;
    a.split_bits = s.split == 4 ? 2 : s.split == 2 ? 1 : 0;
    a.front = plan.r_front;
    a.pitch = plan.r_pitch;
    a.aligned = a.L % 4 == 0 && (reinterpret_cast<uintptr_t>(a.X) & 15u) == 0;
    const size_t bytes = (size_t)(resident_floats(plan, s.examples, a.C) + resident_merge_floats(plan, s.examples, s.parts, s.split, mode)) * sizeof(float);
    const int bands = mode == 2 ? plan.r_back : plan.r_bands;
    auto of = [bands](auto k0, auto k1, auto k2) { return bands == 0 ? k0 : bands == 1 ? k1 : k2; };
    auto kernel = mode == 0   ? of(fast_resident<0, 0>, fast_resident<0, 1>, fast_resident<0, 2>)
                  : mode == 1 ? of(fast_resident<1, 0>, fast_resident<1, 1>, fast_resident<1, 2>)
                  : mode == 3 ? of(fast_resident<3, 0>, fast_resident<3, 1>, fast_resident<3, 2>)
                              : bands == 3 ? fast_resident<2, 3> : bands == 4 ? fast_resident<2, 4> : bands == 5 ? fast_resident<2, 5> : fast_resident<2, 6>;
    kernel<<<s.grid, 32 * resident_warps(mode, bands), bytes, stream>>>(a);
    count_launch();
}

}  // namespace fast
}  // namespace rocket
