// Device helpers shared by the fused kernels (rocket_fast_fwd.cu, rocket_stream.cu): packed arithmetic, the inner loops,
// pooling, barriers and bulk copies, the arguments of a pass.
#pragma once

#include <cfloat>
#include <climits>
#include <cstdint>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

namespace rocket {
namespace fast {

struct FwdArgs {
    PlanDevice plan;
    const float* X;
    int* feat_i;
    unsigned long long* ws;  // soft mode: (fixed-point sum, max key and index) per (example, kernel)
    float c1, c0;            // soft mode: lambda * log2 e, -shift * log2 e
    int N, C, L, K;
    // backward
    const float* dfeat;      // [N][2K]
    const int32_t* argmax;   // [N][K]
    long long* accfix;       // fixed-point sums: dW ragged [n_weights], then db [K]
    const double* scale;     // [K] fixed-point scale of every kernel's sums
    long long n_weights;
    float lambda;
    long long x_row_stride;  // floats between the channel rows of X (L, or the pitch of the zero-margined copy)
    // S kernel: tiles [s_end[i - 1], s_end[i]) are staged for s_examples[i] examples together, as s_groups[i] groups
    int s_end[3], s_examples[3], s_groups[3];
};

// The stream kernel over a pass of f.N examples (rocket_stream.cu); mode: 0 = hard, 1 = soft, 2 = backward, 3 = hard in half
// precision.
void launch_stream(const FwdArgs& f, int mode, int sms, int64_t l2_bytes, bool after_s, cudaStream_t stream);   // after_s: directly behind the S kernel
cudaError_t set_stream_attributes();   // opts the kernel into its shared-memory size

// The resident kernel over N examples (rocket_resident.cu), modes as above.
struct ResidentArgs {
    const RUnit* units;
    const KRec* krec;
    const float* X;
    const uint8_t* X8;       // or raw 8-bit samples, scaled with norm
    NormArgs norm;
    float* feat;
    int32_t* argmax;         // soft: where the maxima are (or null)
    float c1, c0, lambda;
    int N, C, L, K, n_units;
    int examples, groups, parts, run, split_bits;
    int front, pitch;        // floats in front of the first channel row in shared memory, and from row to row
    bool aligned;            // the rows of X start at 16-byte boundaries
    const float* dfeat;      // backward
    const int32_t* argmax_in;
    long long* accfix;
    const double* scale;
    long long n_weights;
};
void launch_resident(ResidentArgs& a, const PlanHost& plan, int mode, int sms, cudaStream_t stream);
cudaError_t set_resident_attributes(int bands, bool backward);

// A launch that may begin while its predecessor in the stream ends (programmatic dependent launch): the kernel itself waits for the
// predecessor with dependency_wait() before it touches anything, or states why it need not.
template <typename... P, typename... A>
inline void launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

namespace {

// Waits until the kernels before this one in the stream are complete and their results visible.
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream begin once every block has come here.
__device__ __forceinline__ void dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

typedef unsigned long long u64;
constexpr unsigned kFull = 0xffffffffu;
constexpr long long kWaitLimitClocks = 1ll << 31;  // about a second: no wait inside a kernel lasts longer

__device__ __forceinline__ u64 pack2(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(u64& acc, u64 a, u64 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ u64 fma2_to(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Order-preserving map float -> signed int (for atomicMax) and back.
__device__ __forceinline__ int float_key(float v) {
    const int b = __float_as_int(v);
    return b >= 0 ? b : b ^ 0x7fffffff;
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

// One channel of one warp tile: 16 output rows of the thread's column pair, 16+ELL-1 input pairs
// streamed past them.  Row s of the tile sits at st[off[s & 3] + (s >> 2) * STEP]; w2 holds the
// channel's negated weights, each twice.  With WIN, only the groups of four rows [gl, gh) are read
// and multiplied (the others hold no sample and are not in shared memory); gl and gh are the same
// for the whole warp.  With FIRST the accumulators come in undefined and every one of them starts as
// init + w[0] * x (its first product), which is bit for bit what starting at init and adding gives.
template <int ELL, int STEP, bool WIN, bool FIRST = false, int R = kR>
__device__ __forceinline__ void conv_channel(const float* __restrict__ st, const int (&off)[4],
                                             const float* __restrict__ w2, u64 (&acc)[R], int gl = 0, int gh = 0,
                                             u64 init = 0ull) {
    static_assert(!(WIN && FIRST), "a windowed pass may skip an accumulator's first product");
    // A warp loads its weights once, lane j weight j, and hands them round: loads of every weight by every lane are ELL more trips
    // through shared memory per channel.  The loop alone went from 94 to 104 multiply-adds/clk/SM at length 9 and 16 rows, from 98
    // to 108 at 24 rows; the hard transform of 60 x 20 x 50,000 from 60.1 to 56.9 ms.
    u64 wp[ELL];
    {
        const int lane = threadIdx.x & 31;
        const float mine = w2[2 * (lane < ELL ? lane : 0)];
#pragma unroll
        for (int j = 0; j < ELL; ++j) {
            const float w = __shfl_sync(kFull, mine, j);
            wp[j] = pack2(w, w);
        }
    }
#pragma unroll
    for (int g = 0; g < (R + ELL - 1 + 3) / 4; ++g) {
        if (!WIN || (g >= gl && g < gh)) {
#pragma unroll
            for (int s = 4 * g; s < 4 * g + 4 && s < R + ELL - 1; ++s) {
                const float* p = st + off[s & 3] + (s >> 2) * STEP;
                const u64 x = *reinterpret_cast<const u64*>(p);
#pragma unroll
                for (int j = 0; j < ELL; ++j) {
                    const int o = s - j;
                    if (o >= 0 && o < R) {
                        if (FIRST && j == 0) acc[o] = fma2_to(wp[0], x, init);
                        else fma2(acc[o], wp[j], x);
                    }
                }
            }
        }
    }
}

// ---- half precision (mode 3): binary16 samples, weights and bias, every multiply-add rounded once to binary16 ----
typedef uint32_t h2;   // two binary16 numbers: the thread's column pair
__device__ __forceinline__ h2 to_h2(float lo, float hi) {   // round to nearest even, both halves
    h2 r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ void hfma2(h2& acc, h2 a, h2 b) {
    asm("fma.rn.f16x2 %0, %1, %2, %0;" : "+r"(acc) : "r"(a), "r"(b));
}
// The pair as two floats (exact); a negative zero (a tiny negative result rounded to zero) becomes +0, so that
// the sign bit means "below zero" as it does for the FP32 accumulators.
__device__ __forceinline__ u64 h2_to_pair(h2 v) {
    asm("add.rn.f16x2 %0, %0, %1;" : "+r"(v) : "r"(0u));
    unsigned short lo, hi;
    asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(v));
    float a, b;
    asm("cvt.f32.f16 %0, %1;" : "=f"(a) : "h"(lo));
    asm("cvt.f32.f16 %0, %1;" : "=f"(b) : "h"(hi));
    return pack2(a, b);
}
// conv_channel in half precision: the FP32 samples of the staged tile and the FP32 weights of the record are
// rounded to binary16 on the way (the same value every time it is used), the accumulators hold 0 - z as binary16.
template <int ELL, int STEP, bool WIN, int R>
__device__ __forceinline__ void conv_channel_h(const float* __restrict__ st, const int (&off)[4],
                                               const float* __restrict__ w2, h2 (&acc)[R], int gl = 0, int gh = 0) {
    h2 wp[ELL];
#pragma unroll
    for (int j = 0; j < ELL; ++j) {
        const float2 v = *reinterpret_cast<const float2*>(w2 + 2 * j);
        wp[j] = to_h2(v.x, v.y);
    }
#pragma unroll
    for (int g = 0; g < (R + ELL - 1 + 3) / 4; ++g) {
        if (!WIN || (g >= gl && g < gh)) {
#pragma unroll
            for (int s = 4 * g; s < 4 * g + 4 && s < R + ELL - 1; ++s) {
                const float2 xf = *reinterpret_cast<const float2*>(st + off[s & 3] + (s >> 2) * STEP);
                const h2 x = to_h2(xf.x, xf.y);
#pragma unroll
                for (int j = 0; j < ELL; ++j) {
                    const int o = s - j;
                    if (o >= 0 && o < R) hfma2(acc[o], wp[j], x);
                }
            }
        }
    }
}
// The accumulators of a tile in half precision start at 0 - bias (rounded to binary16; +0 when it rounds to zero).
template <int R>
__device__ __forceinline__ void init_acc_h(h2 (&acc)[R], float negb) {
    h2 v = to_h2(negb, negb);
    if ((v & 0x7fff7fffu) == 0u) v = 0u;
#pragma unroll
    for (int o = 0; o < R; ++o) acc[o] = v;
}
template <int R>
__device__ __forceinline__ void widen_acc(const h2 (&acch)[R], u64 (&acc)[R]) {
#pragma unroll
    for (int o = 0; o < R; ++o) acc[o] = h2_to_pair(acch[o]);
}

// Adds the PPV count of the thread's 2 x 16 outputs to cnt and folds their min(-z) into mn.  Outputs outside the kernel's range
// never need a test here: their accumulators start at +inf and stay there (sign bit clear,
// neutral for the min).
template <int R>
__device__ __forceinline__ void pool_hard(const u64 (&acc)[R], int& cnt, float& mn) {
    unsigned signs = 0;  // one sign bit per output, shifted in from the right (counted every 16 rows)
#pragma unroll
    for (int o = 0; o < R; ++o) {
        float a, b;
        unpack2(acc[o], a, b);
        signs = __funnelshift_l(__float_as_uint(a), signs, 1);
        signs = __funnelshift_l(__float_as_uint(b), signs, 1);
        mn = min3(mn, a, b);
        if ((o & 15) == 15 && o + 1 < R) { cnt += __popc(signs); signs = 0; }
    }
    cnt += __popc(signs);
}

// The same for a warp tile with outputs that do not exist: m0 / m1 hold one bit per row of the thread's two
// columns (bit o set: row o is an output); the others are replaced by +inf on the way (sign bit clear, neutral
// for the min), so the accumulators may hold anything there.
template <int R>
__device__ __forceinline__ void pool_hard_masked(const u64 (&acc)[R], unsigned m0, unsigned m1, int& cnt, float& mn) {
    const float inf = __int_as_float(0x7f800000);
    unsigned signs = 0;
#pragma unroll
    for (int o = 0; o < R; ++o) {
        float a, b;
        unpack2(acc[o], a, b);
        a = (m0 & (1u << o)) ? a : inf;
        b = (m1 & (1u << o)) ? b : inf;
        signs = __funnelshift_l(__float_as_uint(a), signs, 1);
        signs = __funnelshift_l(__float_as_uint(b), signs, 1);
        mn = min3(mn, a, b);
        if ((o & 15) == 15 && o + 1 < R) { cnt += __popc(signs); signs = 0; }
    }
    cnt += __popc(signs);
}
// Bit o set for lo <= o < hi (0 <= lo, hi <= 31).
__device__ __forceinline__ unsigned row_mask(int lo, int hi) { return hi > lo ? ((1u << hi) - 1u) & ~((1u << lo) - 1u) : 0u; }

// Accumulators of a tile: 0 - bias where the output exists, +inf elsewhere.
template <int R>
__device__ __forceinline__ void init_acc(u64 (&acc)[R], float negb, bool interior, int lo0, int hi0, int lo1, int hi1) {
    if (interior) {
        const u64 v = pack2(negb, negb);
#pragma unroll
        for (int o = 0; o < R; ++o) acc[o] = v;
    } else {
        const float inf = __int_as_float(0x7f800000);
#pragma unroll
        for (int o = 0; o < R; ++o) acc[o] = pack2((o >= lo0 && o < hi0) ? negb : inf, (o >= lo1 && o < hi1) ? negb : inf);
    }
}

__device__ __forceinline__ void publish(int* __restrict__ feat_i, int64_t pair, int cnt, float mn, int lane) {
    cnt = __reduce_add_sync(kFull, cnt);
    const int key = __reduce_max_sync(kFull, float_key(-mn));
    if (lane == 0) {
        if (cnt) atomicAdd(feat_i + pair * 2, cnt);
        atomicMax(feat_i + pair * 2 + 1, key);
    }
}

__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float ex2_approx(float v) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

constexpr float kSoftFixedScale = 1073741824.0f;  // 2^30: soft sums travel as fixed-point integers

// Soft pooling of a warp tile (Eq. 3-4): sum of h = 1 / (1 + 2^(c1 * acc + c0)) over the valid
// outputs (acc = -z, c1 = lambda * log2 e, c0 = -shift * log2 e), the max and the lowest output
// index attaining it.  base0 / base1 are the output indices of row 0 of the thread's two columns,
// step the index distance between rows.  The warp's sum is added to ws[2 * pair] as a fixed-point
// integer and (max key, INT_MAX - index) is folded into ws[2 * pair + 1] with one 64-bit atomic max:
// both are exact and order-free, so results are run-to-run identical.
template <int R>
__device__ __forceinline__ void pool_publish_soft(unsigned long long* __restrict__ ws, int64_t pair, const u64 (&acc)[R],
                                                  float c1, float c0, bool interior, int lo0, int hi0, int lo1, int hi1,
                                                  int base0, int base1, int step, int lane) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f);
    u64 hs = pack2(0.0f, 0.0f);
    float mn = __int_as_float(0x7f800000);
#pragma unroll
    for (int o = 0; o < R; ++o) {
        u64 t = c0p;
        fma2(t, acc[o], c1p);
        float ta, tb, a, b;
        unpack2(t, ta, tb);
        const u64 den = add2(pack2(ex2_approx(ta), ex2_approx(tb)), one);
        unpack2(den, ta, tb);
        float ha = rcp_approx(ta), hb = rcp_approx(tb);
        if (!interior) {
            if (o < lo0 || o >= hi0) ha = 0.0f;
            if (o < lo1 || o >= hi1) hb = 0.0f;
        }
        hs = add2(hs, pack2(ha, hb));
        unpack2(acc[o], a, b);
        mn = min3(mn, a, b);
    }
    float h0, h1;
    unpack2(hs, h0, h1);
    float hsum = h0 + h1;
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) hsum += __shfl_xor_sync(kFull, hsum, sh);
    const int key = float_key(-mn);
    const int wkey = __reduce_max_sync(kFull, key);
    int idx = INT_MAX;
    if (key == wkey) {
#pragma unroll
        for (int o = R - 1; o >= 0; --o) {
            float a, b;
            unpack2(acc[o], a, b);
            if (b == mn) idx = min(idx, base1 + o * step);
            if (a == mn) idx = min(idx, base0 + o * step);
        }
    }
    idx = __reduce_min_sync(kFull, idx);
    if (lane == 0) {
        atomicAdd(ws + 2 * pair, __float2ull_rn(hsum * kSoftFixedScale));
        const unsigned long long k64 = ((unsigned long long)((unsigned)wkey ^ 0x80000000u) << 32) |
                                       (unsigned long long)(unsigned)(INT_MAX - idx);
        atomicMax(ws + 2 * pair + 1, k64);
    }
}

__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Backward, first half: turns the accumulators (acc = -z) of a warp tile into
//   gz = gPs * h (1 - h) + gM [output index == argmax],  h = 1 / (1 + 2^(c1 * acc + c0)),
// zero where the output does not exist, and returns the thread's sum of gz (its share of db).
// oA0 / oA1: the row of the thread's first / second column that is the argmax, or -1.
template <int R>
__device__ __forceinline__ float make_gz(u64 (&acc)[R], float c1, float c0, float gPs, float gM, bool interior, int lo0,
                                         int hi0, int lo1, int hi1, int oA0, int oA1) {
    const u64 c1p = pack2(c1, c1), c0p = pack2(c0, c0), one = pack2(1.0f, 1.0f), neg1 = pack2(-1.0f, -1.0f);
    const u64 gp = pack2(gPs, gPs);
    u64 sum = pack2(0.0f, 0.0f);
#pragma unroll
    for (int o = 0; o < R; ++o) {
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
            if (o < lo0 || o >= hi0) ga = 0.0f;
            if (o < lo1 || o >= hi1) gb = 0.0f;
        }
        if (o == oA0) ga += gM;
        if (o == oA1) gb += gM;
        g = pack2(ga, gb);
        acc[o] = g;
        sum = add2(sum, g);
    }
    float s0, s1;
    unpack2(sum, s0, s1);
    return s0 + s1;
}

// Backward, second half, one channel of one warp tile: dw[j] += gz[o] * x[o + j] for the thread's
// column pair (same traversal as conv_channel with the roles of weights and accumulators swapped).
template <int ELL, int STEP, bool WIN, int R = kR, int A = ELL>
__device__ __forceinline__ void grad_channel(const float* __restrict__ st, const int (&off)[4], const u64 (&gz)[R],
                                             u64 (&dw)[A], int gl = 0, int gh = 0) {
#pragma unroll
    for (int g = 0; g < (R + ELL - 1 + 3) / 4; ++g) {
        if (!WIN || (g >= gl && g < gh)) {
#pragma unroll
            for (int s = 4 * g; s < 4 * g + 4 && s < R + ELL - 1; ++s) {
                const float* p = st + off[s & 3] + (s >> 2) * STEP;
                const u64 x = *reinterpret_cast<const u64*>(p);
#pragma unroll
                for (int j = 0; j < ELL; ++j) {
                    const int o = s - j;
                    if (o >= 0 && o < R) fma2(dw[j], gz[o], x);
                }
            }
        }
    }
}

// Adds a float to a fixed-point accumulator (value * scale as a 64-bit integer): exact and order-free.
__device__ __forceinline__ void add_fixed(long long* dst, float v, double scale) {
    atomicAdd(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)__double2ll_rn((double)v * scale));
}

// Sums dw[j] (both halves) over the warp and adds the ELL totals to dst[0..ELL).  A butterfly that
// halves the number of live values at every step leaves total j on the lanes with (lane >> 1) == j.
template <int ELL>
__device__ __forceinline__ void reduce_publish_dw(const u64 (&dw)[ELL], long long* dst, double scale, int lane, int len = ELL) {
    float v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (j < ELL) {
            float a, b;
            unpack2(dw[j], a, b);
            v[j] = a + b;
        } else {
            v[j] = 0.0f;
        }
    }
#pragma unroll
    for (int half = 8; half >= 1; half >>= 1) {
        const int mask = half * 2;
        const bool up = (lane & mask) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = up ? v[i] : v[i + half];
            const float keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, send, mask);
        }
    }
    const float total = v[0] + __shfl_xor_sync(kFull, v[0], 1);
    const int j = lane >> 1;
    if ((lane & 1) == 0 && j < len) add_fixed(dst + j, total, scale);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
// Wait on a phase parity, bounded in time: returns false when the limit is reached (the caller
// records it and the block winds down).  Between polls the warp sleeps, so a waiting warp does
// not take issue slots from the warps that compute.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        __nanosleep(64);
        if (mbar_try(bar, parity)) return true;
        if (clock64() - t0 > kWaitLimitClocks) return false;
    }
}
// Bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16), completion on bar.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Tiled TMA load of one 4-D box (x a multiple of 4 floats), completion on bar.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, int x, int y, int z, int w, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}

}  // namespace
}  // namespace fast
}  // namespace rocket
