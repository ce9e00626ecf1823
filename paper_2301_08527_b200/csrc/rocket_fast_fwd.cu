// Fused forward kernels of the fast path (hard PPV + max, soft PPV + max + argmax): see rocket_fast.h
// for the geometry.
//
// Arithmetic conventions shared by both kernels
//   - Accumulators hold -z: weights and bias are stored negated (acc = (0 - b) + sum (-w) x).  Then
//     z > 0  <=>  the sign bit of acc is set, exactly: a zero accumulator is always +0 (it starts
//     at +0 when b == 0, exact cancellation rounds to +0, and +0 plus a -0 product stays +0), so
//     the PPV count is one shift-and-add per output and MAX = -min(acc).
//   - A thread's two columns travel together as one packed pair (fma.rn.f32x2 gives each half the
//     result of a separate fused multiply-add).
//   - Outputs outside the kernel's range are replaced by +inf before pooling (sign bit clear,
//     neutral for the min).
//   - Per (example, kernel) the count is combined with integer atomic adds and the max with an
//     integer atomic max on an order-preserving key, both exact and order-independent, so the
//     result is run-to-run identical.  The feature buffer itself holds these integers until the
//     finalise kernel turns them into (count / L_out, max).
#include <cuda.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <mutex>

#include "rocket_fast.h"
#include "rocket_fast_dev.cuh"
#include "rocket_fast_geom.h"

namespace rocket {
namespace fast {
namespace {

extern __shared__ __align__(128) unsigned char smem_raw[];

// ------------------------------------------------------------------------------------------------
// S regime
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, int bytes) {   // bytes: 4, or 0 for a zero
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Backward second half for one kernel on an S tile: per channel, dW sums of the warp tile.  One instance of the reduction for all
// lengths: the code that the warps of an SM run at a time decides how long the backward waits for instructions.
template <int R>
__device__ __forceinline__ void s_grad_tile(const float* planes, const KRec* rec, int len, int lane, const u64 (&gz)[R], long long* accfix,
                                            double scale) {
    const int m = __shfl_sync(kFull, rec->m, 0);
    const int off[4] = {2 * lane, kWarpCols + 2 * lane, 2 * kWarpCols + 2 * lane, 3 * kWarpCols + 2 * lane};
    for (int q = 0; q < m; ++q) {
        u64 dw[ROCKET_MAX_LENGTH];
#pragma unroll
        for (int j = 0; j < ROCKET_MAX_LENGTH; ++j) dw[j] = 0ull;
        const float* st = planes + rec->ch[q] * s_plane_floats(R);
        if (len == 7) grad_channel<7, 4 * kWarpCols, false, R>(st, off, gz, dw);
        else if (len == 9) grad_channel<9, 4 * kWarpCols, false, R>(st, off, gz, dw);
        else grad_channel<11, 4 * kWarpCols, false, R>(st, off, gz, dw);
        reduce_publish_dw<ROCKET_MAX_LENGTH>(dw, accfix + rec->woff + q * len, scale, lane, len);
    }
}

// The channels of one kernel on an S tile.  fold: the accumulators come in undefined and start at the
// kernel's 0 - bias inside the first channel's pass (every output of the warp tile exists).
template <int ELL, bool FOLD, int R>
__device__ __forceinline__ void s_kernel_tile(const float* planes, const KRec* rec, int lane, u64 (&acc)[R]) {
    const int m = __shfl_sync(kFull, rec->m, 0);
    const int off[4] = {2 * lane, kWarpCols + 2 * lane, 2 * kWarpCols + 2 * lane, 3 * kWarpCols + 2 * lane};
    int q = 0;
    if constexpr (FOLD) {
        const float nb = rec->negb;
        conv_channel<ELL, 4 * kWarpCols, false, true, R>(planes + rec->ch[0] * s_plane_floats(R), off, rec->w2[0], acc, 0, 0, pack2(nb, nb));
        q = 1;
    }
    for (; q < m; ++q)
        conv_channel<ELL, 4 * kWarpCols, false, false, R>(planes + rec->ch[q] * s_plane_floats(R), off, rec->w2[q], acc);
}

// The same in half precision (mode 3).
template <int ELL, int R>
__device__ __forceinline__ void s_kernel_tile_h(const float* planes, const KRec* rec, int lane, h2 (&acc)[R]) {
    const int m = __shfl_sync(kFull, rec->m, 0);
    const int off[4] = {2 * lane, kWarpCols + 2 * lane, 2 * kWarpCols + 2 * lane, 3 * kWarpCols + 2 * lane};
    for (int q = 0; q < m; ++q)
        conv_channel_h<ELL, 4 * kWarpCols, false, R>(planes + rec->ch[q] * s_plane_floats(R), off, rec->w2[q], acc);
}

// Bound: the packed multiply-adds of the inner loops (78 % of a tile's time at dilations below 8), and for the larger dilations, where
// a bucket has few kernels, what a tile costs besides: 2,600 clocks to draw it, 7,400 (dilations 32 to 63) to 20,000 (dilation 1,
// whose columns are 24 samples apart) to copy it in - the lines an SM can have in flight, about 24 B/clk, whether the copies are
// asynchronous, plain loads in batches or 16 bytes wide - and 800 to 5,400 that the warps wait for the last kernel; of 27,000 clocks
// at dilations 32 to 63, 11,400 are work.  Measured at 60 x 20 x 50,000, hard: 24.1 ms with weights read by every lane, 22.6 now.
// Tried and not kept: two half tiles in flight behind producer warps (22.9 ms; 22 input rows for 12 rows of outputs make the
// shared memory the limit), drawing the next tile during the copies (22.5 to 22.6, and late draws matter for small batches).
template <int MODE, int ROWS = kRS, bool HALF = false>  // 0 = hard, 1 = soft, 2 = backward of soft, 3 = hard in half precision; ROWS: of a band; HALF: a wide handle
__global__ void __launch_bounds__(kSThreads, 1) fast_s_forward(FwdArgs a) {
    dependency_wait();
    // The stream kernel needs what came before this one, not this one: it may begin on the SMs that run out of tiles (8 x 20 x 10,001:
    // 1.52 -> 1.45 ms; 10 x 6 x 1,251, 1,000 kernels: soft transform 88 -> 72 us).
    dependency_release();
    constexpr int R = HALF ? kSHalfRows : ROWS, kPlanes = HALF ? kSWidePlanes : kSMaxPlanes, kPlaneFloats = s_plane_floats(R);
    float* planes = reinterpret_cast<float*>(smem_raw);                               // [kPlanes][rows][64]
    KRec* recs = reinterpret_cast<KRec*>(planes + kPlanes * kPlaneFloats);             // [warps][2]
    __shared__ unsigned s_item;
    __shared__ int s_next, s_n0, s_ne, s_half;
    __shared__ SItem s_sitem;
    __shared__ SBucket s_bucket;
    __shared__ long long s_src[kPlanes];      // where the planes' channel rows start in X
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // Work is handed out as (tile, group of examples), the tiles of the buckets with many kernels first.  Where a bucket has
    // few kernels, several examples share a tile's planes, as far as they fit: the warps then find (kernel, example) pairs
    // enough to keep busy.
    const unsigned tiles0 = (unsigned)a.s_end[0] * (unsigned)a.s_groups[0], tiles1 = (unsigned)(a.s_end[1] - a.s_end[0]) * (unsigned)a.s_groups[1];
    const unsigned total = (tiles0 + tiles1 + (unsigned)(a.s_end[2] - a.s_end[1]) * (unsigned)a.s_groups[2]) * (HALF ? 2u : 1u);
    KRec* myrec = recs + warp * 2;

    bool first = true;
    for (;;) {
        __syncthreads();  // the previous tile is fully consumed
        if (warp == 0) {  // draw a tile and lay its description out for the block
            unsigned g = 0;
            if (first) g = blockIdx.x;            // a block's first tile goes by its place, which spares a trip to the counter
            else if (lane == 0) g = gridDim.x + atomicAdd(a.plan.counters + 0, 1u);
            g = __shfl_sync(kFull, g, 0);
            first = false;
            if (lane == 0) { s_item = g; s_next = 0; }
            if (g < total) {
                if (HALF) {
                    if (lane == 0) s_half = (int)(g & 1u);
                    g >>= 1;
                }
                const int cls = g < tiles0 ? 0 : g < tiles0 + tiles1 ? 1 : 2;
                const unsigned first = cls == 0 ? 0u : (unsigned)a.s_end[cls - 1], count = (unsigned)a.s_end[cls] - first;
                const unsigned rest = g - (cls == 0 ? 0u : cls == 1 ? tiles0 : tiles0 + tiles1);
                const int n0 = (int)(rest / count) * a.s_examples[cls], ne = min(a.s_examples[cls], a.N - n0);
                if (lane == 0) { s_n0 = n0; s_ne = ne; }
                const SItem it = a.plan.sitems[first + rest % count];
                const SBucket* __restrict__ src = a.plan.sb + it.bucket;
                if (lane == 0) s_sitem = it;
                if (lane < kSBucketWords) reinterpret_cast<int*>(&s_bucket)[lane] = __ldg(reinterpret_cast<const int*>(src) + lane);
                const int nch = __ldg(&src->nch);
                auto plane_src = [&](int pl) {
                    const int e = pl / nch;
                    if (e < ne) s_src[pl] = ((long long)(n0 + e) * a.C + __ldg(&src->ch[pl - e * nch])) * a.x_row_stride;
                };
                plane_src(lane);
                if (HALF) plane_src(lane + 32);
            }
        }
        __syncthreads();
        if (s_item >= total) break;
        const int n0 = s_n0, ne = s_ne;
        const SItem item = s_sitem;
        const SBucket& b = s_bucket;
        const int d = b.d, kbeg = b.kbeg, n_work = (b.kend - kbeg) * ne, nch = b.nch;
        const bool tile_interior = item.interior != 0;
        const int half_row = HALF ? s_half * R : 0;              // the first row of the half

        // Stage the tile: every plane, rows 0..rows-1 of every column, zero outside the series.  A thread takes one column of
        // every eighth row; what does not depend on the plane is computed once, so that a sample costs an address and a copy.
        {
            constexpr int kStep = kSThreads / kWarpCols, kRows = (R + ROCKET_MAX_LENGTH - 1 + kStep - 1) / kStep;
            const int col = threadIdx.x & (kWarpCols - 1), rg = threadIdx.x / kWarpCols;
            const int cg = item.c0 + col;
            const bool col_ok = cg < b.raster_len;
            const int fu0 = s_column_u0(b, cg, ROWS) + half_row * d, n_planes = nch * ne, rows = b.rows - (ROWS - R);
            int xi[kRows], bytes[kRows];
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const int s = rg + i * kStep, x = fu0 + s * d;
                const bool ok = col_ok && s < rows && (unsigned)x < (unsigned)a.L;
                xi[i] = ok ? x : 0;
                bytes[i] = ok ? 4 : 0;
            }
            uint32_t dst = smem_u32(planes + rg * kWarpCols + col);
#pragma unroll 4
            for (int c = 0; c < n_planes; ++c) {
                const float* __restrict__ src = a.X + s_src[c];
#pragma unroll
                for (int i = 0; i < kRows; ++i)
                    if (rg + i * kStep < rows) cp_async4(dst + i * kStep * kWarpCols * 4, src + xi[i], bytes[i]);
                dst += kPlaneFloats * 4;
            }
            cp_async_commit();
        }
        // the thread's two columns
        const int cg0 = item.c0 + 2 * lane;
        const bool ok0 = cg0 < b.raster_len, ok1 = cg0 + 1 < b.raster_len;
        const int band0 = cg0 / d, c0 = cg0 - band0 * d;          // (first A-row, residue) of the two columns
        const int band1 = c0 + 1 < d ? band0 : band0 + 1, c1 = c0 + 1 < d ? c0 + 1 : 0;
        const int trow0 = b.tmin + band0 * ROWS + half_row, trow1 = b.tmin + band1 * ROWS + half_row;
        cp_async_wait<0>();
        __syncthreads();

        // (kernel, example) pairs of the bucket, pulled from the shared counter, kernel by kernel; the record of the next
        // one is copied into the warp's other slot while the current one computes
        const unsigned inv_ne = (65536u + (unsigned)ne - 1u) / (unsigned)ne;   // several examples only with fewer than 32 kernels
        auto kernel_of = [&](int w) { return ne == 1 ? w : (int)(((unsigned)w * inv_ne) >> 16); };
        auto fetch = [&](int w, int slot) {
            if (w < n_work) {
                const char* src = reinterpret_cast<const char*>(a.plan.krec + kbeg + kernel_of(w));
                const uint32_t dst = smem_u32(myrec + slot);
                for (int i = lane; i < (int)(sizeof(KRec) / 16); i += 32) cp_async16(dst + 16 * i, src + 16 * i);
            }
            cp_async_commit();
        };
        int kk = 0;
        if (lane == 0) kk = atomicAdd(&s_next, 1);
        kk = __shfl_sync(kFull, kk, 0);
        int cur = 0;
        fetch(kk, cur);
        while (kk < n_work) {
            int kk_next = 0;
            if (lane == 0) kk_next = atomicAdd(&s_next, 1);
            kk_next = __shfl_sync(kFull, kk_next, 0);
            fetch(kk_next, cur ^ 1);
            cp_async_wait<1>();
            __syncwarp();
            const int example = ne == 1 ? 0 : kk - kernel_of(kk) * ne, n = n0 + example;
            const float* eplanes = planes + example * nch * kPlaneFloats;   // the example's planes
            const KRec* rec = myrec + cur;
            // the same for the warp: as a shuffle's result the compiler takes it for uniform and keeps the branches on it cheap
            const int len = __shfl_sync(kFull, rec->len, 0), korig = rec->k;
            // on an interior tile (the plan's flag) every output exists for every kernel of the bucket
            int lo0 = 0, hi0 = R, lo1 = 0, hi1 = R;
            bool interior = tile_interior;
            if (!tile_interior) {
                valid_rows_tc(trow0, c0, rec->tl, rec->rl, rec->th, rec->rh, R, ok0, lo0, hi0);
                valid_rows_tc(trow1, c1, rec->tl, rec->rl, rec->th, rec->rh, R, ok1, lo1, hi1);
                interior = __all_sync(kFull, lo0 == 0 && lo1 == 0 && hi0 == R && hi1 == R);
            }
            u64 acc[R];
            // hard mode: the pooling masks the outputs that do not exist, so the accumulators always start inside
            // the first channel's pass; the other modes start them at 0 - bias, or +inf where there is no output
            constexpr bool kFold = MODE == 0;
            if constexpr (MODE == 3) {
                h2 acch[R];
                init_acc_h(acch, rec->negb);
                if (len == 7) s_kernel_tile_h<7>(eplanes, rec, lane, acch);
                else if (len == 9) s_kernel_tile_h<9>(eplanes, rec, lane, acch);
                else s_kernel_tile_h<11>(eplanes, rec, lane, acch);
                widen_acc(acch, acc);
            } else {
                if (!kFold) init_acc(acc, rec->negb, interior, lo0, hi0, lo1, hi1);
                if (len == 7) s_kernel_tile<7, kFold>(eplanes, rec, lane, acc);
                else if (len == 9) s_kernel_tile<9, kFold>(eplanes, rec, lane, acc);
                else s_kernel_tile<11, kFold>(eplanes, rec, lane, acc);
            }
            if (MODE == 2) {
                const int64_t pair = (int64_t)n * a.K + korig;
                const float gP = __ldg(a.dfeat + 2 * pair), gM = __ldg(a.dfeat + 2 * pair + 1);
                const int uA = __ldg(a.argmax + pair) - rec->p;
                int tA = uA / d, cA = uA - tA * d;                        // floor division: uA >= -p may be negative
                if (cA < 0) { cA += d; --tA; }
                const int oA0 = (ok0 && c0 == cA && tA >= trow0 && tA < trow0 + R) ? tA - trow0 : -1;
                const int oA1 = (ok1 && c1 == cA && tA >= trow1 && tA < trow1 + R) ? tA - trow1 : -1;
                float dbs = make_gz(acc, a.c1, a.c0, gP * a.lambda / (float)rec->nout, gM, interior, lo0, hi0, lo1, hi1, oA0, oA1);
#pragma unroll
                for (int sh = 16; sh > 0; sh >>= 1) dbs += __shfl_xor_sync(kFull, dbs, sh);
                const double scale = __ldg(a.scale + korig);
                if (lane == 0) add_fixed(a.accfix + a.n_weights + korig, dbs, scale);
                s_grad_tile(eplanes, rec, len, lane, acc, a.accfix, scale);
            } else if (MODE == 1) {
                const int p = rec->p;
                pool_publish_soft(a.ws, (int64_t)n * a.K + korig, acc, a.c1, a.c0, interior, lo0, hi0, lo1, hi1,
                                  trow0 * d + c0 + p, trow1 * d + c1 + p, d, lane);
            } else {
                int cnt = 0;
                float mn = __int_as_float(0x7f800000);
                if (interior) pool_hard(acc, cnt, mn);
                else pool_hard_masked(acc, row_mask(lo0, hi0), row_mask(lo1, hi1), cnt, mn);
                publish(a.feat_i, (int64_t)n * a.K + korig, cnt, mn, lane);
            }
            __syncwarp();  // every lane is done with the record before its slot is refilled
            kk = kk_next;
            cur ^= 1;
        }
        cp_async_wait<0>();
    }
}

// ------------------------------------------------------------------------------------------------
// T regime
// ------------------------------------------------------------------------------------------------
// What the producer tells the consumers about a tile (written with plain stores before its
// arrive on the stage's barrier, which releases them).
struct TSlotItem {
    int32_t t0, r0, rg, cg, box_rows, rec_slot, wide, g_lo;
    int32_t g_hi, n, stop, flags;         // n: example of the tile; stop: no tile, the block is done;
                                          // flags: the plan's warp_interior | warp_active << 8
};

// Dynamic shared memory of one group: the stages of its ring, then its kernel-record slots (a multiple of 128 bytes).
constexpr size_t kTGroupSmemBytes = ((size_t)kTStages * kTStageFloats * 4 + (size_t)kTParamSlots * sizeof(KRec) + 127) / 128 * 128;

struct TShared {
    unsigned long long full[kTStages];
    unsigned long long empty[kTStages];
    TSlotItem items[kTParamSlots];
    int abort;
};

// The channels of one tile for one consumer warp; returns false when a wait gave up.  A warp
// without a valid output (active == false) only keeps the ring moving.
template <int ELL, int STEP, bool WIN>
__device__ __forceinline__ bool t_channels(const float* stages, const KRec* rec, const int (&off)[4], uint32_t full0,
                                           uint32_t empty0, uint32_t& st, int lane, bool active, u64 (&acc)[kR], int gl,
                                           int gh) {
    const int m = rec->m;
    for (int q = 0; q < m; ++q) {
        const uint32_t slot = st % kTStages;
        if (q > 0 && !mbar_wait(full0 + 8u * slot, (st / kTStages) & 1u)) return false;
        if (active) conv_channel<ELL, STEP, WIN>(stages + slot * kTStageFloats, off, rec->w2[q], acc, gl, gh);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8u * slot);
        ++st;
    }
    return true;
}

// Backward second half on a T tile: the kernel's channels stream through the ring once more.
template <int ELL, int STEP, bool WIN>
__device__ __forceinline__ bool t_grad_channels(const float* stages, const KRec* rec, const int (&off)[4], uint32_t full0,
                                                uint32_t empty0, uint32_t& st, int lane, bool active, const u64 (&gz)[kR],
                                                long long* accfix, double scale, int gl, int gh) {
    const int m = rec->m;
    for (int q = 0; q < m; ++q) {
        const uint32_t slot = st % kTStages;
        if (!mbar_wait(full0 + 8u * slot, (st / kTStages) & 1u)) return false;
        if (active) {
            u64 dw[ELL];
#pragma unroll
            for (int j = 0; j < ELL; ++j) dw[j] = 0ull;
            grad_channel<ELL, STEP, WIN>(stages + slot * kTStageFloats, off, gz, dw, gl, gh);
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + 8u * slot);
            reduce_publish_dw<ELL>(dw, accfix + rec->woff + q * ELL, scale, lane);
        } else {
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + 8u * slot);
        }
        ++st;
    }
    return true;
}

template <int STEP, bool WIN>
__device__ __forceinline__ bool t_grad_dispatch(int len, const float* stages, const KRec* rec, const int (&off)[4],
                                                uint32_t full0, uint32_t empty0, uint32_t& st, int lane, bool active,
                                                const u64 (&gz)[kR], long long* accfix, double scale, int gl, int gh) {
    if (len == 7) return t_grad_channels<7, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, gz, accfix, scale, gl, gh);
    if (len == 9) return t_grad_channels<9, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, gz, accfix, scale, gl, gh);
    return t_grad_channels<11, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, gz, accfix, scale, gl, gh);
}

template <int STEP, bool WIN>
__device__ __forceinline__ bool t_dispatch(int len, const float* stages, const KRec* rec, const int (&off)[4],
                                           uint32_t full0, uint32_t empty0, uint32_t& st, int lane, bool active,
                                           u64 (&acc)[kR], int gl, int gh) {
    if (len == 7) return t_channels<7, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
    if (len == 9) return t_channels<9, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
    return t_channels<11, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
}

// The channels of one tile in half precision (mode 3).
template <int ELL, int STEP, bool WIN>
__device__ __forceinline__ bool t_channels_h(const float* stages, const KRec* rec, const int (&off)[4], uint32_t full0,
                                             uint32_t empty0, uint32_t& st, int lane, bool active, h2 (&acc)[kR], int gl,
                                             int gh) {
    const int m = rec->m;
    for (int q = 0; q < m; ++q) {
        const uint32_t slot = st % kTStages;
        if (q > 0 && !mbar_wait(full0 + 8u * slot, (st / kTStages) & 1u)) return false;
        if (active) conv_channel_h<ELL, STEP, WIN, kR>(stages + slot * kTStageFloats, off, rec->w2[q], acc, gl, gh);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8u * slot);
        ++st;
    }
    return true;
}
template <int STEP, bool WIN>
__device__ __forceinline__ bool t_dispatch_h(int len, const float* stages, const KRec* rec, const int (&off)[4],
                                             uint32_t full0, uint32_t empty0, uint32_t& st, int lane, bool active,
                                             h2 (&acc)[kR], int gl, int gh) {
    if (len == 7) return t_channels_h<7, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
    if (len == 9) return t_channels_h<9, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
    return t_channels_h<11, STEP, WIN>(stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
}

template <int MODE>  // 0 = hard, 1 = soft, 2 = backward of soft, 3 = hard in half precision
__global__ void __launch_bounds__(kTBlockThreads, kTBlocksPerSM) fast_t_forward(FwdArgs a) {
    __shared__ __align__(16) TShared shs[kTGroups];
    // the block's groups work independently of one another: each has its part of the shared memory
    const int group = threadIdx.x / kTThreads, tid = threadIdx.x - group * kTThreads;
    TShared& sh = shs[group];
    // dynamic shared memory, aligned to 128 bytes by hand: per group its stages, then its kernel-record slots
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* base = smem_raw + (((raw + 127u) & ~127u) - raw) + (size_t)group * kTGroupSmemBytes;
    float* stages = reinterpret_cast<float*>(base);
    KRec* recs = reinterpret_cast<KRec*>(base + (size_t)kTStages * kTStageFloats * 4);
    const int lane = tid & 31, warp = tid >> 5;
    const uint32_t full0 = smem_u32(sh.full), empty0 = smem_u32(sh.empty);
    if (tid == 0) {
        for (int i = 0; i < kTStages; ++i) {
            mbar_init(full0 + 8u * i, 1);
            mbar_init(empty0 + 8u * i, kTConsumerWarps);
        }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // Work is handed out in units of kTChunkTiles consecutive tiles of one example, example after
    // example (all blocks read one example at a time, so it stays in L2; consecutive tiles mostly
    // share a kernel).  The producer draws the units from a global counter and tells the consumers
    // what to do through the ring, a stop item last.
    const unsigned n_chunks = ((unsigned)a.plan.n_titems + kTChunkTiles - 1u) / kTChunkTiles;
    const unsigned total_units = (unsigned)a.N * n_chunks;
    volatile int* abort_flag = &sh.abort;

    if (warp == kTConsumerWarps) {
        // ---- producer: one lane issues every copy of the block
        if (lane == 0) {
            uint32_t st = 0, it = 0, nrec = 0;
            int cur_krec = -1;
            bool ok = true;
            unsigned u = atomicAdd(a.plan.counters + 1, 1u);
            while (ok && u < total_units) {
                const unsigned u_next = atomicAdd(a.plan.counters + 1, 1u);   // on its way while this unit is issued
                const int n = (int)(u / n_chunks);
                const int i_beg = (int)((u - (unsigned)n * n_chunks) * kTChunkTiles);
                const int i_end = min(i_beg + (int)kTChunkTiles, a.plan.n_titems);
                const int4* tp = reinterpret_cast<const int4*>(a.plan.titems + i_beg);
                int4 w0 = __ldg(tp), w1 = __ldg(tp + 1), w2 = __ldg(tp + 2), w3 = __ldg(tp + 3), w4 = __ldg(tp + 4),
                     w5 = __ldg(tp + 5), w6 = __ldg(tp + 6), w7 = __ldg(tp + 7);
                for (int i = i_beg; ok && i < i_end; ++i) {
                    if (*abort_flag) { ok = false; break; }
                    const int map = w0.x, t0 = w0.y, r0 = w0.z, rg = w0.w;
                    const int m = w1.z, box_rows = w1.w, krec = w2.w, cg = w3.x, wide = w3.y, g_lo = w3.z, g_hi = w3.w;
                    const unsigned chw[3] = {(unsigned)w2.x, (unsigned)w2.y, (unsigned)w2.z};
                    const int px[4] = {w4.x, w4.y, w4.z, w4.w}, py[4] = {w5.x, w5.y, w5.z, w5.w}, pj[4] = {w6.x, w6.y, w6.z, w6.w};
                    const int run = 4 * w1.x;
                    const int flags = (w7.x & 0xff) | ((w7.y & 0xff) << 8);
                    {   // the next tile's description is on its way while this one is issued
                        const int inext = min(i + 1, i_end - 1);
                        tp = reinterpret_cast<const int4*>(a.plan.titems + inext);
                        w0 = __ldg(tp); w1 = __ldg(tp + 1); w2 = __ldg(tp + 2); w3 = __ldg(tp + 3); w4 = __ldg(tp + 4);
                        w5 = __ldg(tp + 5); w6 = __ldg(tp + 6); w7 = __ldg(tp + 7);
                    }
                    const uint32_t box_bytes = (uint32_t)box_rows * (uint32_t)t_box_cols(cg) * 4u;
                    const uint32_t phase_bytes = (uint32_t)t_phase_floats(cg, box_rows) * 4u;
                    const char* tmap = reinterpret_cast<const char*>(a.plan.tmaps) + (size_t)map * 128;
                    const bool new_rec = krec != cur_krec;
                    if (new_rec) { cur_krec = krec; ++nrec; }
                    const uint32_t rslot = (nrec - 1u) % kTParamSlots;
                    const int n_stages = MODE == 2 ? 2 * m : m;   // the backward streams the channels twice
                    for (int q2 = 0; q2 < n_stages; ++q2) {
                        const int q = q2 < m ? q2 : q2 - m;
                        const uint32_t slot = st % kTStages;
                        if (st >= (uint32_t)kTStages && !mbar_wait(empty0 + 8u * slot, ((st / kTStages) - 1u) & 1u)) {
                            ok = false;
                            break;
                        }
                        const uint32_t bar = full0 + 8u * slot;
                        uint32_t tx = (wide ? 4u * (uint32_t)kTWideHalves : 4u) * box_bytes;
                        if (q2 == 0) {
                            TSlotItem& si = sh.items[it % kTParamSlots];
                            si.t0 = t0; si.r0 = r0; si.rg = rg; si.cg = cg; si.box_rows = box_rows; si.rec_slot = (int)rslot;
                            si.wide = wide; si.g_lo = g_lo; si.g_hi = g_hi; si.n = n; si.stop = 0; si.flags = flags;
                            if (new_rec) tx += (uint32_t)sizeof(KRec);
                        }
                        mbar_arrive_expect_tx(bar, tx);
                        if (q2 == 0 && new_rec) bulk_g2s(smem_u32(recs + rslot), a.plan.krec + krec, (uint32_t)sizeof(KRec), bar);
                        const int ch = (int)((chw[q >> 2] >> (8 * (q & 3))) & 0xffu);
                        const int z = n * a.C + ch;
                        const uint32_t dst0 = smem_u32(stages + slot * kTStageFloats);
#pragma unroll
                        for (int k = 0; k < 4; ++k) tma_load_4d(dst0 + (uint32_t)k * phase_bytes, tmap, px[k], py[k], z, pj[k], bar);
                        if (wide) {   // the further halves: the boxes 256 columns further right each
                            for (int h = 1; h < kTWideHalves; ++h) {
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    int x2 = px[k] + h * kTWideCols, y2 = py[k];
                                    while (x2 >= run) { x2 -= run; ++y2; }
                                    tma_load_4d(dst0 + (uint32_t)(4 * h + k) * phase_bytes, tmap, x2, y2, z, pj[k], bar);
                                }
                            }
                        }
                        ++st;
                    }
                    ++it;
                }
                u = u_next;
            }
            if (ok) {   // the stop item takes a stage of its own (no copy)
                const uint32_t slot = st % kTStages;
                if (st >= (uint32_t)kTStages && !mbar_wait(empty0 + 8u * slot, ((st / kTStages) - 1u) & 1u)) {
                    ok = false;
                } else {
                    sh.items[it % kTParamSlots].stop = 1;
                    mbar_arrive(full0 + 8u * slot);
                    ++st;
                }
            }
            if (!ok) {
                *abort_flag = 1;
                atomicExch(a.plan.error_flag, 1);
            }
            // nothing of this block may still be in flight when it exits: every issued stage has
            // either been consumed or is waited for here (bounded)
            for (uint32_t back = 1; back <= (uint32_t)kTStages && back <= st; ++back) {
                const uint32_t s2 = st - back;
                mbar_wait(full0 + 8u * (s2 % kTStages), (s2 / kTStages) & 1u);
            }
        }
    } else {
        // ---- consumers
        uint32_t st = 0, it = 0;
        bool ok = true;
        // hard mode: the count and the min(-z) of the (example, kernel) pair the warp is working on travel from
        // tile to tile (consecutive tiles mostly share a kernel) and are published when the pair changes
        int64_t cur_pair = -1;
        int cnt = 0;
        float mn = __int_as_float(0x7f800000);
        for (;;) {
            if (*abort_flag) { ok = false; break; }
            const uint32_t slot = st % kTStages;
            if (!mbar_wait(full0 + 8u * slot, (st / kTStages) & 1u)) {
                ok = false;
                break;
            }
            const TSlotItem si = sh.items[it % kTParamSlots];
            if (si.stop) break;
            const int n = si.n;
            const KRec* rec = recs + si.rec_slot;
            const int t0 = si.t0, r0 = si.r0, cg = si.cg, box_rows = si.box_rows;
            const int len = rec->len, d = rec->d, korig = rec->k;
            const bool wide = si.wide != 0;
            // warp tile (wr, wc) of the tile; a wide tile is one row of all consumer warps' tiles
            const int wr = wide ? 0 : (cg == 1 ? warp : (cg == 2 ? warp >> 1 : warp >> 2));
            const int wc = wide ? warp : (warp & (cg - 1));
            const int lc = kWarpCols * wc + 2 * lane;
            // the plan says per warp whether every / any output of its warp tile exists
            bool interior = ((si.flags >> warp) & 1) != 0;
            const bool active = ((si.flags >> (8 + warp)) & 1) != 0;
            const bool ok0 = active && r0 + lc < d, ok1 = active && r0 + lc + 1 < d;
            int lo0 = 0, hi0 = kR, lo1 = 0, hi1 = kR;
            if (active && !interior) {
                valid_rows_tc(t0 + kR * wr, r0 + lc, rec->tl, rec->rl, rec->th, rec->rh, kR, ok0, lo0, hi0);
                valid_rows_tc(t0 + kR * wr, r0 + lc + 1, rec->tl, rec->rl, rec->th, rec->rh, kR, ok1, lo1, hi1);
            }
            // where rows 0..3 of the warp tile sit in a stage: the box of phase k starts k * phase floats in; an
            // ordinary tile's warp tile starts 4 wr box rows down, a wide tile's in half lc / 256, g_lo box rows up
            // (t_elem_offset / t_wide_elem_offset for tile rows 0..3)
            const int boxw = wide ? kTWideCols : t_box_cols(cg);
            const int phase = box_rows * boxw;
            const int base = wide ? (lc >> 8) * (4 * phase) - si.g_lo * kTWideCols + (lc & (kTWideCols - 1)) : 4 * wr * boxw + lc;
            const int off[4] = {base, base + phase, base + 2 * phase, base + 3 * phase};
            const int gl = si.g_lo, gh = si.g_hi;
            u64 acc[kR];
            // Hard mode: every accumulator starts at 0 - bias and the pooling masks the outputs that do not exist.
            // The other modes start at +inf where there is no output.  (Starting the accumulators inside the first
            // channel's pass, as the small-dilation kernel does, doubles the inner-loop instances here: measured
            // slower, the kernel then waits for instructions.)
            if constexpr (MODE == 3) {
                h2 acch[kR];
                init_acc_h(acch, rec->negb);
                if (wide) ok = t_dispatch_h<kTWideCols, true>(len, stages, rec, off, full0, empty0, st, lane, active, acch, gl, gh);
                else if (cg == 1) ok = t_dispatch_h<kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acch, 0, 0);
                else if (cg == 2) ok = t_dispatch_h<2 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acch, 0, 0);
                else ok = t_dispatch_h<4 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acch, 0, 0);
                widen_acc(acch, acc);
            } else {
                if (active) init_acc(acc, rec->negb, interior || MODE == 0, lo0, hi0, lo1, hi1);
                if (wide) ok = t_dispatch<kTWideCols, true>(len, stages, rec, off, full0, empty0, st, lane, active, acc, gl, gh);
                else if (cg == 1) ok = t_dispatch<kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, 0, 0);
                else if (cg == 2) ok = t_dispatch<2 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, 0, 0);
                else ok = t_dispatch<4 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, 0, 0);
            }
            if (!ok) break;
            const int64_t pair = (int64_t)n * a.K + korig;
            if (MODE == 2) {
                double scale = 0.0;
                if (active) {
                    const float gP = __ldg(a.dfeat + 2 * pair), gM = __ldg(a.dfeat + 2 * pair + 1);
                    const int uA = __ldg(a.argmax + pair) - rec->p;
                    int tA = uA / d, cA = uA - tA * d;                        // floor division: uA >= -p may be negative
                    if (cA < 0) { cA += d; --tA; }
                    const int trow = t0 + kR * wr, c0 = r0 + lc;
                    const bool rowhit = tA >= trow && tA < trow + kR;
                    const int oA0 = (ok0 && rowhit && c0 == cA) ? tA - trow : -1;
                    const int oA1 = (ok1 && rowhit && c0 + 1 == cA) ? tA - trow : -1;
                    float dbs = make_gz(acc, a.c1, a.c0, gP * a.lambda / (float)rec->nout, gM, interior, lo0, hi0, lo1, hi1, oA0,
                                        oA1);
#pragma unroll
                    for (int sh = 16; sh > 0; sh >>= 1) dbs += __shfl_xor_sync(kFull, dbs, sh);
                    scale = __ldg(a.scale + korig);
                    if (lane == 0) add_fixed(a.accfix + a.n_weights + korig, dbs, scale);
                }
                if (wide) ok = t_grad_dispatch<kTWideCols, true>(len, stages, rec, off, full0, empty0, st, lane, active, acc, a.accfix, scale, gl, gh);
                else if (cg == 1) ok = t_grad_dispatch<kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, a.accfix, scale, 0, 0);
                else if (cg == 2) ok = t_grad_dispatch<2 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, a.accfix, scale, 0, 0);
                else ok = t_grad_dispatch<4 * kWarpCols, false>(len, stages, rec, off, full0, empty0, st, lane, active, acc, a.accfix, scale, 0, 0);
                if (!ok) break;
            } else if (active) {
                if (MODE == 1) {
                    const int base = (t0 + kR * wr) * d + r0 + lc + rec->p;
                    pool_publish_soft(a.ws, pair, acc, a.c1, a.c0, interior, lo0, hi0, lo1, hi1, base, base + 1, d, lane);
                } else {
                    if (pair != cur_pair) {
                        if (cur_pair >= 0) publish(a.feat_i, cur_pair, cnt, mn, lane);
                        cur_pair = pair;
                        cnt = 0;
                        mn = __int_as_float(0x7f800000);
                    }
                    if (interior) pool_hard(acc, cnt, mn);
                    else pool_hard_masked(acc, row_mask(lo0, hi0), row_mask(lo1, hi1), cnt, mn);
                }
            }
            ++it;
        }
        // what the warp still carries is published even when a wait gave up: counts and maxima are only
        // ever combined with commutative atomics, and the error flag marks the result as incomplete
        if ((MODE == 0 || MODE == 3) && cur_pair >= 0) publish(a.feat_i, cur_pair, cnt, mn, lane);
        if (!ok) {
            *abort_flag = 1;
            if (lane == 0) atomicExch(a.plan.error_flag, 1);
        }
    }
    __syncthreads();  // every wait above is bounded, so every warp gets here
}

// ------------------------------------------------------------------------------------------------
// pad copy / init / finalise
// ------------------------------------------------------------------------------------------------
// Writes the samples of the batch into the four shifted copies: copy j holds the zero-margined
// layout moved down by j floats (copy_j[i] = layout[i + j]); margins are never written and stay zero.
__global__ void fast_pad_copy_kernel(const float4* __restrict__ X, float* __restrict__ xpad, int64_t rows, int L4,
                                     int64_t pitch, int front, int64_t copy_floats) {
    const int64_t total = rows * L4;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = e / L4;
        const int i = (int)(e - rho * L4);
        const float4 v = __ldg(X + e);
        float* dst = xpad + rho * pitch + front + 4 * (int64_t)i;
        *reinterpret_cast<float4*>(dst) = v;
#pragma unroll
        for (int j = 1; j < 4; ++j) {
            float* dj = dst + j * copy_floats - j;
            dj[0] = v.x; dj[1] = v.y; dj[2] = v.z; dj[3] = v.w;
        }
    }
}

// The same for series whose length is not a multiple of four floats, or whose base is not 16-byte aligned:
// one float per thread and step.
__global__ void fast_pad_copy_scalar_kernel(const float* __restrict__ X, float* __restrict__ xpad, int64_t rows, int L,
                                            int64_t pitch, int front, int64_t copy_floats) {
    const int64_t total = rows * L;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = e / L;
        const int i = (int)(e - rho * L);
        const float v = __ldg(X + e);
        float* dst = xpad + rho * pitch + front + i;
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[j * copy_floats - j] = v;
    }
}

// The same from raw 8-bit intensities (Section 4.1): every sample becomes (v - mean[c]) * inv_std[c]
// (per-channel feature scaling, Section 4.3) on its way into the four copies.
__global__ void fast_pad_copy_u8_kernel(const uchar4* __restrict__ X, float* __restrict__ xpad, int64_t rows, int L4,
                                        int C, int64_t pitch, int front, int64_t copy_floats, NormArgs norm) {
    const int64_t total = rows * L4;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = e / L4;
        const int i = (int)(e - rho * L4);
        const int c = (int)(rho % C);
        const uchar4 u = __ldg(X + e);
        const float mu = norm.mean[c], is = norm.inv_std[c];
        float4 v;
        v.x = ((float)u.x - mu) * is; v.y = ((float)u.y - mu) * is;
        v.z = ((float)u.z - mu) * is; v.w = ((float)u.w - mu) * is;
        float* dst = xpad + rho * pitch + front + 4 * (int64_t)i;
        *reinterpret_cast<float4*>(dst) = v;
#pragma unroll
        for (int j = 1; j < 4; ++j) {
            float* dj = dst + j * copy_floats - j;
            dj[0] = v.x; dj[1] = v.y; dj[2] = v.z; dj[3] = v.w;
        }
    }
}

// The seven shifted copies of the stream kernel: copy j of a channel row holds the row moved down by j floats.  A thread writes
// floats 4 i .. 4 i + 3 of every copy from ten samples; i runs from -2 (samples that the shift brings below the row's start)
// and zeros are written past its end.
template <typename Load>
__device__ __forceinline__ void write_stream_copies(float* __restrict__ row0, int64_t pitch, int front, int i4, int L, Load&& load) {
    float v[12];
    load(v);
#pragma unroll
    for (int e = 0; e < 10; ++e)
        if ((unsigned)(4 * i4 + e) >= (unsigned)L) v[e] = 0.0f;
#pragma unroll
    for (int j = 0; j < kWCopies; ++j)
        *reinterpret_cast<float4*>(row0 + j * pitch + front + 4 * i4) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
}
template <bool VEC>   // VEC: rows start at 16-byte boundaries
__global__ void stream_copy_kernel(const float* __restrict__ X, float* __restrict__ wpad, int64_t rows, int L, int64_t pitch, int front) {
    dependency_wait();
    const int per = (L + 3) / 4 + 2;
    const int64_t total = rows * per;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = e / per;
        const int i4 = (int)(e - rho * per) - 2;
        const float* __restrict__ x = X + rho * L;
        write_stream_copies(wpad + rho * kWCopies * pitch, pitch, front, i4, L, [&](float (&v)[12]) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int at = 4 * (i4 + q);
                if (VEC) {
                    const float4 f = at >= 0 && at < L ? __ldg(reinterpret_cast<const float4*>(x + at)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[4 * q + c] = at + c >= 0 && at + c < L ? __ldg(x + at + c) : 0.0f;
                }
            }
        });
    }
}
__global__ void stream_copy_u8_kernel(const uint8_t* __restrict__ X, float* __restrict__ wpad, int64_t rows, int L, int C, int64_t pitch,
                                      int front, NormArgs norm) {
    const int per = (L + 3) / 4 + 2;
    const int64_t total = rows * per;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rho = e / per;
        const int i4 = (int)(e - rho * per) - 2, ch = (int)(rho % C);
        const float mu = norm.mean[ch], is = norm.inv_std[ch];
        const uint8_t* __restrict__ x = X + rho * L;
        write_stream_copies(wpad + rho * kWCopies * pitch, pitch, front, i4, L, [&](float (&v)[12]) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int at = 4 * (i4 + q);   // L and the base are multiples of four
                const uchar4 u = at >= 0 && at < L ? __ldg(reinterpret_cast<const uchar4*>(x + at)) : make_uchar4(0, 0, 0, 0);
                v[4 * q] = ((float)u.x - mu) * is; v[4 * q + 1] = ((float)u.y - mu) * is;
                v[4 * q + 2] = ((float)u.z - mu) * is; v[4 * q + 3] = ((float)u.w - mu) * is;
            }
        });
    }
}

__global__ void fast_init_kernel(int* __restrict__ feat_i, int64_t pairs, unsigned* counters) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e == 0) { counters[0] = 0u; counters[1] = 0u; }
    if (e < pairs) { feat_i[2 * e] = 0; feat_i[2 * e + 1] = INT_MIN; }
}

__global__ void fast_finalize_kernel(float* __restrict__ feat, const KRec* __restrict__ krec, int n_krec, int N,
                                     int K) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)N * n_krec) return;
    const int n = (int)(e / n_krec), f = (int)(e - (int64_t)n * n_krec);
    const int k = krec[f].k, nout = krec[f].nout;
    int* fi = reinterpret_cast<int*>(feat) + ((int64_t)n * K + k) * 2;
    const int cnt = fi[0], key = fi[1];
    feat[((int64_t)n * K + k) * 2] = (float)cnt / (float)nout;   // Eq. 2
    feat[((int64_t)n * K + k) * 2 + 1] = key_float(key);
}

__global__ void fast_init_soft_kernel(unsigned long long* __restrict__ ws, int64_t pairs, unsigned* counters) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e == 0) { counters[0] = 0u; counters[1] = 0u; }
    if (e < pairs) { ws[2 * e] = 0ull; ws[2 * e + 1] = 0ull; }
}

__global__ void fast_finalize_soft_kernel(float* __restrict__ feat, int32_t* __restrict__ argmax,
                                          const unsigned long long* __restrict__ ws, const KRec* __restrict__ krec,
                                          int n_krec, int N, int K) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)N * n_krec) return;
    const int n = (int)(e / n_krec), f = (int)(e - (int64_t)n * n_krec);
    const int k = krec[f].k, nout = krec[f].nout;
    const int64_t pair = (int64_t)n * K + k;
    const unsigned long long sum = ws[2 * pair], k64 = ws[2 * pair + 1];
    feat[pair * 2] = (float)((double)sum / (double)kSoftFixedScale / (double)nout);   // Eq. 4
    feat[pair * 2 + 1] = key_float((int)((unsigned)(k64 >> 32) ^ 0x80000000u));
    if (argmax) argmax[pair] = INT_MAX - (int)(unsigned)(k64 & 0xffffffffull);
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

size_t s_smem_bytes(bool wide) {
    return (size_t)(wide ? kSWidePlanes * s_plane_floats(kSHalfRows) : kSMaxPlanes * kSPlaneFloats) * 4 + (size_t)kSWarps * 2 * sizeof(KRec);
}
size_t t_smem_bytes() { return (size_t)kTGroups * kTGroupSmemBytes + 128; }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

template <typename... K>
cudaError_t allow_smem(size_t bytes, K... kernels) {
    cudaError_t e = cudaSuccess;
    ((e = e == cudaSuccess ? cudaFuncSetAttribute(kernels, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : e), ...);
    return e;
}
template <int ROWS>
cudaError_t allow_s() {
    return allow_smem(s_smem_bytes(false), fast_s_forward<0, ROWS>, fast_s_forward<1, ROWS>, fast_s_forward<2, ROWS>, fast_s_forward<3, ROWS>);
}
// Opts the fused kernels that a handle's calls may launch into their dynamic shared memory sizes, once per device and kind of kernel (which
// also loads them: all kinds take milliseconds).
cudaError_t set_kernel_attributes(int dev, const PlanHost& h) {
    static std::mutex attr_mu;
    std::lock_guard<std::mutex> attr_lock(attr_mu);
    static bool done_for[64][13] = {};
    bool* done = done_for[dev & 63];
    cudaError_t e = cudaSuccess;
    auto once = [&](int kind, bool needed, auto&& set) {
        if (e != cudaSuccess || done[kind] || !needed) return;
        e = set();
        done[kind] = e == cudaSuccess;
    };
    for (int bands = 0; bands < 3; ++bands) once(6 + bands, h.resident && h.r_bands == bands, [bands] { return set_resident_attributes(bands, false); });
    for (int bands : kRBackBands) once(6 + bands, h.r_back == bands, [bands] { return set_resident_attributes(bands, true); });
    once(0, !h.sitems.empty() && !h.s_wide && h.s_rows == kRS, allow_s<kRS>);
    once(1, !h.sitems.empty() && h.s_rows == kSLowRows[0], allow_s<kSLowRows[0]>);
    once(2, !h.sitems.empty() && h.s_rows == kSLowRows[1], allow_s<kSLowRows[1]>);
    once(3, h.s_wide, [] { return allow_smem(s_smem_bytes(true), fast_s_forward<0, kRS, true>, fast_s_forward<1, kRS, true>, fast_s_forward<2, kRS, true>); });
    once(4, !h.wunits.empty(), [] { return set_stream_attributes(); });
    once(5, !h.titems.empty(), [] { return allow_smem(t_smem_bytes(), fast_t_forward<0>, fast_t_forward<1>, fast_t_forward<2>, fast_t_forward<3>); });
    return e;
}

// ---- backward helpers ----------------------------------------------------------------------------
// Largest |x| of the batch, as the bit pattern of a non-negative float (integer order = float order).  One atomic per block of 256
// threads: one per warp, all to the same word, took 8 us of a minibatch.
__device__ __forceinline__ unsigned block_max(float m) {
    __shared__ unsigned s_max;
    if (threadIdx.x == 0) s_max = 0u;
    __syncthreads();
    const unsigned b = __reduce_max_sync(kFull, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, b);
    __syncthreads();
    return s_max;
}
__global__ void fast_absmax_scalar_kernel(const float* __restrict__ X, int64_t n, unsigned* __restrict__ out) {
    float m = 0.0f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(__ldg(X + e)));
    const unsigned b = block_max(m);
    if (threadIdx.x == 0) atomicMax(out, b);
}

__global__ void fast_absmax_kernel(const float4* __restrict__ X, int64_t n4, unsigned* __restrict__ out) {
    float m = 0.0f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n4; e += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = __ldg(X + e);
        m = fmaxf(fmaxf(m, fabsf(v.x)), fmaxf(fabsf(v.y), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
    const unsigned b = block_max(m);
    if (threadIdx.x == 0) atomicMax(out, b);
}

// Per kernel: a bound on sum |gz| |x| over the batch gives the fixed-point scale of its sums
// (|sum_i gz_i| <= |gP| lambda / 4 + |gM| per example since h (1 - h) <= 1/4), and its sums are cleared.  A warp per kernel here
// and in the finalise kernel: a thread per kernel went through up to 121 weights one by one (8 and 13 us of a minibatch).
// Of a batch of at most kSmallBatch samples every block takes the maximum itself (small: the batch), which spares clearing the word and a launch.
constexpr int64_t kSmallBatch = 4096;
__global__ void fast_bwd_prepare_kernel(const float* __restrict__ dfeat, const KRec* __restrict__ krec, int n_krec, int N,
                                        int K, float lambda, const unsigned* __restrict__ absmax_bits, const float* __restrict__ small, int n_small,
                                        double* __restrict__ scale, long long* __restrict__ accfix, long long n_weights,
                                        unsigned* __restrict__ counters) {
    unsigned most = 0u;
    if (small) {
        float m = 0.0f;
#pragma unroll 8
        for (int e = threadIdx.x; e < n_small; e += blockDim.x) m = fmaxf(m, fabsf(__ldg(small + e)));
        most = block_max(m);
    }
    dependency_wait();
    const int f = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (f >= n_krec) return;
    const KRec& r = krec[f];
    const int k = r.k, taps = r.m * r.len;
    double bound = 0.0;
    for (int n = lane; n < N; n += 32) {
        const float gP = __ldg(dfeat + ((int64_t)n * K + k) * 2), gM = __ldg(dfeat + ((int64_t)n * K + k) * 2 + 1);
        bound += (double)fabsf(gP) * (double)fabsf(lambda) * 0.25 + (double)fabsf(gM);
    }
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) bound += __shfl_xor_sync(kFull, bound, sh);
    for (int t = lane; t < taps; t += 32) accfix[r.woff + t] = 0;
    if (lane > 0) return;
    const double xmax = fmax((double)__uint_as_float(small ? most : *absmax_bits), 1.0);
    bound *= xmax * 1.01;
    scale[k] = (bound > 0.0 && bound < 1e300) ? 1152921504606846976.0 / bound : 0.0;  // 2^60 / bound
    accfix[n_weights + k] = 0;
    if (f == 0) { counters[0] = 0u; counters[1] = 0u; }
}

__global__ void fast_bwd_finalize_kernel(const long long* __restrict__ accfix, const double* __restrict__ scale,
                                         const KRec* __restrict__ krec, int n_krec, long long n_weights,
                                         float* __restrict__ dW, float* __restrict__ db) {
    const int f = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (f >= n_krec) return;
    const KRec& r = krec[f];
    const int k = r.k, taps = r.m * r.len;
    const double sc = scale[k], inv = sc > 0.0 ? 1.0 / sc : 0.0;
    for (int t = lane; t < taps; t += 32) dW[r.woff + t] = (float)((double)accfix[r.woff + t] * inv);
    if (lane == 0) db[k] = (float)((double)accfix[n_weights + k] * inv);
}

}  // namespace

// Examples per pass through the fused kernels: as many as keep the staging copies of a pass at kWCopyBytes (13 of 20 x 50,000),
// or near what 12 examples of that size take in the four-copy form; passes of few short series would end in launches with
// nothing to do for most SMs.  Without copies one pass does.
static int chunk_examples(const FastState& fs, int C, bool stream, bool copies) {
    if (stream) return stream_chunk(C, fs.host.wpitch);
    if (!copies) return 1 << 16;
    return (int)std::max<int64_t>(kChunkExamples, 80000000ll / (4 * (int64_t)C * fs.host.pad_pitch));
}

// The S tiles of a pass (mode: 0 = hard, 1 = soft, 2 = backward, 3 = hard in half precision, whose series are never wide).
// after_kernel: what comes before it in the stream is a kernel of this call (a programmatic launch depends on nothing else).
static void launch_s(FwdArgs& a, const FastState& fs, int mode, int sms, bool after_kernel, cudaStream_t stream) {
    const SGroups share = s_groups(fs.host, a.N, sms);
    for (int cls = 0; cls < 3; ++cls) {
        a.s_end[cls] = share.end[cls];
        a.s_examples[cls] = share.examples[cls];
        a.s_groups[cls] = share.groups[cls];
    }
    const unsigned grid = share.grid;
    const bool wide = fs.host.s_wide;
    const size_t bytes = s_smem_bytes(wide);
    auto launch = [&](auto kernel) {
        if (after_kernel) launch_dependent(kernel, grid, kSThreads, bytes, stream, a);
        else kernel<<<grid, kSThreads, bytes, stream>>>(a);
    };
    auto rows = [&](auto mode_tag) {
        constexpr int MODE = decltype(mode_tag)::value;
        if (wide && MODE != 3) launch(fast_s_forward<MODE, kRS, MODE != 3>);
        else if (fs.host.s_rows == kSLowRows[0]) launch(fast_s_forward<MODE, kSLowRows[0]>);
        else if (fs.host.s_rows == kSLowRows[1]) launch(fast_s_forward<MODE, kSLowRows[1]>);
        else launch(fast_s_forward<MODE>);
    };
    if (mode == 0) rows(std::integral_constant<int, 0>{});
    else if (mode == 1) rows(std::integral_constant<int, 1>{});
    else if (mode == 2) rows(std::integral_constant<int, 2>{});
    else rows(std::integral_constant<int, 3>{});
    count_launch();
}

// Blocks of the T kernel: as many as are resident at a time, never more than there are work units.
static unsigned t_grid(int n_examples, int n_titems, int sms) {
    const unsigned long long units = (unsigned long long)n_examples * ((n_titems + kTChunkTiles - 1) / kTChunkTiles);
    return (unsigned)std::min<unsigned long long>((units + kTGroups - 1) / kTGroups, (unsigned long long)kTBlocksPerSM * (unsigned long long)sms);
}

cudaError_t upload_plan(FastState& fs) {
    const PlanHost& h = fs.host;
    PlanDevice& d = fs.dev;
    d = PlanDevice();
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&fs.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&fs.l2_bytes, cudaDevAttrL2CacheSize, dev);
    if (e != cudaSuccess) return e;
    struct Part { const void* src; size_t bytes; size_t off; };
    Part parts[9] = {
        {h.krec.data(), h.krec.size() * sizeof(KRec), 0},   {h.sb.data(), h.sb.size() * sizeof(SBucket), 0},
        {h.sitems.data(), h.sitems.size() * sizeof(SItem), 0}, {h.titems.data(), h.titems.size() * sizeof(TItem), 0},
        {h.generic_list.data(), h.generic_list.size() * 4, 0}, {nullptr, 256, 0}, {nullptr, 256, 0},
        {h.wunits.data(), h.wunits.size() * sizeof(WUnit), 0}, {h.runits.data(), h.runits.size() * sizeof(RUnit), 0}};
    size_t total = 0;
    for (auto& pt : parts) { pt.off = total; total += align256(pt.bytes); }
    e = device_malloc(&fs.plan_blob, std::max<size_t>(total, 256));
    if (e != cudaSuccess) { fs.plan_blob = nullptr; return e; }
    char* base = static_cast<char*>(fs.plan_blob);
    e = cudaMemset(base, 0, std::max<size_t>(total, 256));
    for (auto& pt : parts)
        if (e == cudaSuccess && pt.src && pt.bytes) e = cudaMemcpy(base + pt.off, pt.src, pt.bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { cudaFree(fs.plan_blob); fs.plan_blob = nullptr; return e; }
    d.krec = reinterpret_cast<const KRec*>(base + parts[0].off);
    d.sb = reinterpret_cast<const SBucket*>(base + parts[1].off);
    d.sitems = reinterpret_cast<const SItem*>(base + parts[2].off);
    d.titems = reinterpret_cast<const TItem*>(base + parts[3].off);
    d.generic_list = reinterpret_cast<const int32_t*>(base + parts[4].off);
    d.counters = reinterpret_cast<unsigned*>(base + parts[5].off);
    d.error_flag = reinterpret_cast<int*>(base + parts[6].off);
    d.wunits = reinterpret_cast<const WUnit*>(base + parts[7].off);
    d.runits = reinterpret_cast<const RUnit*>(base + parts[8].off);
    d.n_wunits = (int)h.wunits.size();
    d.w_visits = h.w_visits;
    d.n_krec = (int)h.krec.size(); d.n_sitems = (int)h.sitems.size(); d.n_titems = (int)h.titems.size();
    d.n_generic = (int)h.generic_list.size(); d.n_tmaps = (int)h.tmaps.size();
    d.pad_pitch = h.pad_pitch;
    return cudaSuccess;
}

cudaError_t upload_records(FastState& fs) {
    if (!fs.plan_blob || fs.host.krec.empty()) return cudaSuccess;
    return cudaMemcpy(const_cast<KRec*>(fs.dev.krec), fs.host.krec.data(), fs.host.krec.size() * sizeof(KRec),
                      cudaMemcpyHostToDevice);
}

void release_fast_state(FastState& fs) {
    if (fs.plan_blob) cudaFree(fs.plan_blob);
    if (fs.maps_blob) cudaFree(fs.maps_blob);
    if (fs.xpad) cudaFree(fs.xpad);
    if (fs.wpad) cudaFree(fs.wpad);
    if (fs.wmaps_blob) cudaFree(fs.wmaps_blob);
    if (fs.soft_ws) cudaFree(fs.soft_ws);
    if (fs.bwd_ws) cudaFree(fs.bwd_ws);
    fs.bwd_ws = nullptr;
    fs.soft_ws = nullptr;
    fs.soft_ws_bytes = 0;
    for (cudaEvent_t ev : fs.evs) cudaEventDestroy(ev);
    fs.evs.clear();
    fs.ev_chunks = 0;
    fs.plan_blob = fs.maps_blob = nullptr;
    fs.xpad = fs.wpad = nullptr;
    fs.wmaps_blob = nullptr;
    fs.pad_examples = fs.wpad_examples = 0;
}

// Room for the copies of N examples in place of what *buf holds; N comes back smaller when there is room for fewer, which later
// calls then ask for (a failed allocation of this size takes milliseconds).
template <class Bytes>
static cudaError_t allocate_copies(FastState& fs, float** buf, int& held, int& N, Bytes&& bytes_of) {
    if (*buf) cudaFree(*buf);  // waits for work that still reads it
    *buf = nullptr;
    held = 0;
    cudaError_t e = cudaSuccess;
    const int got = fit_examples(N, [&](int n) {
        e = device_malloc(reinterpret_cast<void**>(buf), bytes_of(n));
        if (e != cudaSuccess) *buf = nullptr;
        return e != cudaErrorMemoryAllocation;
    });
    if (got < N) fs.most_examples = got;
    if (got > 0 && e == cudaSuccess && got < N) cudaGetLastError();   // of the larger sizes
    N = got;
    return e;
}

cudaError_t ensure_stream_capacity(FastState& fs, int N, int C, int L) {
    N = std::min(N, fs.most_examples);
    if (N == 0) return cudaErrorMemoryAllocation;
    if (N <= fs.wpad_examples) return cudaSuccess;
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return cudaErrorNotSupported;
    const int64_t pitch = fs.host.wpitch, front = fs.host.wfront;
    auto bytes_of = [&](int n) { return (size_t)((int64_t)n * C * kWCopies * pitch + front + pitch) * sizeof(float); };   // a box may run past the last copy
    cudaError_t e = allocate_copies(fs, &fs.wpad, fs.wpad_examples, N, bytes_of);
    if (e != cudaSuccess) return e;
    e = cudaMemset(fs.wpad, 0, bytes_of(N));  // the margins stay zero from here on
    if (e != cudaSuccess) return e;
    const int64_t copies = (int64_t)N * C * kWCopies;
    const size_t n_maps = fs.host.wmaps.size();
    std::vector<CUtensorMap> maps(n_maps);
    for (size_t i = 0; i < n_maps; ++i) {
        const WMapSpec& sp = fs.host.wmaps[i];
        const int64_t d = sp.d, G = w_rows_per_y(sp.d), run = G * d;
        // floats from one row of a y step to the next: so many copies on, so many samples on
        const int64_t step = d % 4 == 1 ? pitch + d - 1 : d % 4 == 3 ? pitch - d - 1 : d % 4 == 2 ? 2 * pitch + d - 2 : pitch;
        // y steps that hold samples (counted backwards, a step's first row lies three rows further on)
        const int64_t ny = (front + L + (d % 4 == 3 ? 3 * d : 0) + run - 1) / run;
        const cuuint64_t dims[4] = {(cuuint64_t)(run + kWarpCols), (cuuint64_t)G, (cuuint64_t)ny, (cuuint64_t)copies};
        const cuuint64_t strides[3] = {(cuuint64_t)step * 4u, (cuuint64_t)run * 4u, (cuuint64_t)pitch * 4u};
        const cuuint32_t box[4] = {(cuuint32_t)kWarpCols, (cuuint32_t)G, (cuuint32_t)sp.y_rows, 1u};
        const cuuint32_t elem[4] = {1u, 1u, 1u, 1u};
        const CUresult r = encode(&maps[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, fs.wpad, dims, strides, box, elem,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    if (!fs.wmaps_blob) {
        e = device_malloc(&fs.wmaps_blob, n_maps * sizeof(CUtensorMap));
        if (e != cudaSuccess) { fs.wmaps_blob = nullptr; return e; }
    }
    e = cudaMemcpy(fs.wmaps_blob, maps.data(), n_maps * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    fs.wpad_examples = N;
    fs.dev.wmaps = fs.wmaps_blob;
    return cudaSuccess;
}

// Writes `rows` channel rows of X into the stream kernel's copies.
static void launch_stream_copy(FastState& fs, const float* X, int64_t rows, int L, int sms, bool dependent, cudaStream_t stream) {
    const bool vec = L % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    auto kernel = vec ? stream_copy_kernel<true> : stream_copy_kernel<false>;
    if (dependent) launch_dependent(kernel, sms * 8, 256, 0, stream, X, fs.wpad, rows, L, fs.host.wpitch, (int)fs.host.wfront);
    else kernel<<<sms * 8, 256, 0, stream>>>(X, fs.wpad, rows, L, fs.host.wpitch, (int)fs.host.wfront);
    count_launch();
}

cudaError_t ensure_pad_capacity(FastState& fs, int N, int C, int L, bool without_maps) {
    if (fs.host.tmaps.empty() && !without_maps) return cudaSuccess;
    N = std::min(N, fs.most_examples);
    if (N == 0) return cudaErrorMemoryAllocation;
    if (N <= fs.pad_examples) return cudaSuccess;
    EncodeTiledFn encode = fs.host.tmaps.empty() ? nullptr : encode_tiled_fn();
    if (!encode && !fs.host.tmaps.empty()) return cudaErrorNotSupported;
    const int64_t pitch = fs.host.pad_pitch;          // a multiple of 32 floats
    auto bytes_of = [&](int n) { return (size_t)((int64_t)n * C + 1) * pitch * 4 * 4; };
    cudaError_t e = allocate_copies(fs, &fs.xpad, fs.pad_examples, N, bytes_of);
    if (e != cudaSuccess) return e;
    const int64_t rows = (int64_t)N * C, copy_floats = (rows + 1) * pitch;
    e = cudaMemset(fs.xpad, 0, bytes_of(N));  // the margins stay zero from here on: the pad copy writes samples only
    if (e != cudaSuccess) return e;
    const size_t n_maps = fs.host.tmaps.size();
    std::vector<CUtensorMap> maps(n_maps);
    for (size_t i = 0; i < n_maps; ++i) {
        const TMapSpec& sp = fs.host.tmaps[i];
        const cuuint64_t run = 4ull * (cuuint64_t)sp.d;
        const cuuint64_t dims[4] = {run + kTXExtra, ((cuuint64_t)kTPadFront + (cuuint64_t)L + run - 1) / run, (cuuint64_t)rows, 4ull};
        const cuuint64_t strides[3] = {run * 4ull, (cuuint64_t)pitch * 4ull, (cuuint64_t)copy_floats * 4ull};
        const cuuint32_t box[4] = {(cuuint32_t)sp.box_cols, (cuuint32_t)sp.box_rows, 1u, 1u};
        const cuuint32_t elem[4] = {1u, 1u, 1u, 1u};
        const CUresult r = encode(&maps[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, fs.xpad, dims, strides, box, elem,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    static_assert(sizeof(CUtensorMap) == 128, "tensor maps are addressed in 128-byte steps");
    if (n_maps > 0) {
        if (!fs.maps_blob) {
            e = device_malloc(&fs.maps_blob, n_maps * sizeof(CUtensorMap));
            if (e != cudaSuccess) { fs.maps_blob = nullptr; return e; }
        }
        e = cudaMemcpy(fs.maps_blob, maps.data(), n_maps * sizeof(CUtensorMap), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return e;
    }
    fs.pad_examples = N;
    fs.copy_floats = copy_floats;
    fs.dev.tmaps = fs.maps_blob;
    fs.dev.xpad = fs.xpad;
    return cudaSuccess;
}

// Writes `rows` channel rows of X into the four shifted zero-margined copies (16-byte pieces when the rows allow).
static void launch_pad_copy(FastState& fs, const float* X, int64_t rows, int L, int sms, cudaStream_t stream) {
    if (L % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0)
        fast_pad_copy_kernel<<<sms * 8, 256, 0, stream>>>(reinterpret_cast<const float4*>(X), fs.xpad, rows, L / 4, fs.host.pad_pitch,
                                                          kTPadFront, fs.copy_floats);
    else
        fast_pad_copy_scalar_kernel<<<sms * 8, 256, 0, stream>>>(X, fs.xpad, rows, L, fs.host.pad_pitch, kTPadFront, fs.copy_floats);
    count_launch();
}

// Soft transform: 16 bytes per (example, kernel), grow-only.
static cudaError_t ensure_soft_ws(FastState& fs, int64_t pairs) {
    if ((size_t)pairs * 16 <= fs.soft_ws_bytes) return cudaSuccess;
    if (fs.soft_ws) cudaFree(fs.soft_ws);  // waits for work that still uses it
    fs.soft_ws = nullptr;
    fs.soft_ws_bytes = 0;
    cudaError_t e = device_malloc(&fs.soft_ws, (size_t)pairs * 16);
    if (e != cudaSuccess) { fs.soft_ws = nullptr; return e; }
    fs.soft_ws_bytes = (size_t)pairs * 16;
    return cudaSuccess;
}

// Backward: fixed-point sums [n_weights + K], scales [K], max |x| (fixed size per handle).
static cudaError_t ensure_bwd_ws(FastState& fs, const DeviceParams& dp, int64_t n_weights) {
    if (fs.bwd_ws) return cudaSuccess;
    const size_t acc_bytes = align256((size_t)(n_weights + dp.K) * 8), scale_bytes = align256((size_t)dp.K * 8);
    cudaError_t e = device_malloc(&fs.bwd_ws, acc_bytes + scale_bytes + 256);
    if (e != cudaSuccess) fs.bwd_ws = nullptr;
    return e;
}

// Room for the copies of a hard transform of N examples that the resident kernel could serve as well; that one does where there is none,
// or where making it would end a capture.
static bool tiles_have_room(FastState& fs, const DeviceParams& dp, int N, bool u8, cudaStream_t stream = nullptr) {
    const bool streamed = fs.dev.n_wunits > 0, copies = fs.dev.n_titems > 0 || u8;
    const int n = std::min({N, chunk_examples(fs, dp.C, streamed, copies), fs.most_examples});
    if ((!streamed && !copies) || (n > 0 && n <= (streamed ? fs.wpad_examples : fs.pad_examples))) return true;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = stream ? cudaStreamIsCapturing(stream, &capture) : cudaSuccess;
    if (e == cudaSuccess && capture == cudaStreamCaptureStatusNone)
        e = streamed ? ensure_stream_capacity(fs, n, dp.C, dp.L) : ensure_pad_capacity(fs, n, dp.C, dp.L, u8 && fs.dev.n_titems == 0);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && capture == cudaStreamCaptureStatusNone;
}

cudaError_t reserve_fast_state(FastState& fs, const DeviceParams& dp, int max_N, bool hard, bool soft, bool backward, bool u8,
                               int64_t n_weights, bool again) {
    std::lock_guard<std::mutex> lk(fs.mu);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = set_kernel_attributes(dev, fs.host)) != cudaSuccess) return e;
    if (again) fs.most_examples = 1 << 30;
    if (fs.host.resident && (!backward || resident_backward(fs.host))) {   // no copies, no sums but the backward's
        if (!resident_forward(fs.host, max_N, hard)) tiles_have_room(fs, dp, max_N, u8);
        return backward ? ensure_bwd_ws(fs, dp, n_weights) : cudaSuccess;
    }
    const bool stream = fs.dev.n_wunits > 0, copies = fs.dev.n_titems > 0 || u8;
    const int chunk = std::min(max_N, chunk_examples(fs, dp.C, stream, copies));
    if (stream && (e = ensure_stream_capacity(fs, chunk, dp.C, dp.L)) != cudaSuccess) return e;
    if (!stream && copies && (e = ensure_pad_capacity(fs, chunk, dp.C, dp.L, u8 && fs.dev.n_titems == 0)) != cudaSuccess) return e;
    if (soft && (e = ensure_soft_ws(fs, (int64_t)max_N * dp.K)) != cudaSuccess) return e;
    if (backward && (e = ensure_bwd_ws(fs, dp, n_weights)) != cudaSuccess) return e;
    return cudaSuccess;
}

// What the resident kernel's modes have in common.
static ResidentArgs resident_args(const FastState& fs, const DeviceParams& dp, const float* X, int N, float lambda, float shift) {
    ResidentArgs a{};
    a.units = fs.dev.runits;
    a.n_units = (int)fs.host.runits.size();
    a.krec = fs.dev.krec;
    a.X = X;
    a.c1 = lambda * 1.4426950408889634f; a.c0 = -shift * 1.4426950408889634f; a.lambda = lambda;
    a.N = N; a.C = dp.C; a.L = dp.L; a.K = dp.K;
    return a;
}

cudaError_t launch_fast_forward(FastState& fs, const DeviceParams& dp, const float* X, int N, float* feat,
                                cudaStream_t stream, bool soft, float lambda, float shift, int32_t* argmax,
                                const uint8_t* X_u8, const NormArgs* norm, bool half) {
    if (half && soft) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lk(fs.mu);
    const int sms = fs.sms, l2 = fs.l2_bytes;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = set_kernel_attributes(dev, fs.host);
    if (e != cudaSuccess) return e;
    if (resident_forward(fs.host, N, !soft && !half) || (fs.host.resident && !tiles_have_room(fs, dp, N, X_u8 != nullptr, stream))) {
        ResidentArgs r = resident_args(fs, dp, X, N, lambda, shift);
        r.feat = feat;
        r.argmax = argmax;
        r.X8 = X_u8;
        if (X_u8) r.norm = *norm;
        if (fs.profile) {                                  // one kernel, reported as the small dilations'
            while (fs.evs.size() < 3) {
                cudaEvent_t ev = nullptr;
                if ((e = cudaEventCreate(&ev)) != cudaSuccess) return e;
                fs.evs.push_back(ev);
            }
            cudaEventRecord(fs.evs[0], stream);
        }
        launch_resident(r, fs.host, soft ? 1 : half ? 3 : 0, sms, stream);
        if (fs.profile) {
            cudaEventRecord(fs.evs[1], stream);
            cudaEventRecord(fs.evs[2], stream);
            fs.ev_chunks = 1;
        }
        return cudaGetLastError();
    }
    const size_t t_bytes = t_smem_bytes();
    const PlanDevice& pd = fs.dev;
    // the stream kernel takes the dilations the S kernel leaves; the T kernel where the stream kernel's copies have no room
    const bool streamed = pd.n_wunits > 0, copied = pd.n_titems > 0 || X_u8;
    int chunk = chunk_examples(fs, dp.C, streamed, copied);
    if (streamed) e = ensure_stream_capacity(fs, std::min(N, chunk), dp.C, dp.L);
    else if (copied) e = ensure_pad_capacity(fs, std::min(N, chunk), dp.C, dp.L, X_u8 != nullptr);
    if (e != cudaSuccess) return e;
    if (streamed || copied) chunk = std::min(chunk, fs.most_examples);
    const int64_t pairs = (int64_t)N * dp.K;
    if (soft && (e = ensure_soft_ws(fs, pairs)) != cudaSuccess) return e;
    FwdArgs a;
    a.plan = fs.dev;
    a.c1 = lambda * 1.4426950408889634f; a.c0 = -shift * 1.4426950408889634f;
    a.C = dp.C; a.L = dp.L; a.K = dp.K;
    a.dfeat = nullptr; a.argmax = nullptr; a.accfix = nullptr; a.scale = nullptr; a.n_weights = 0; a.lambda = lambda;
    int* feat_i = reinterpret_cast<int*>(feat);
    unsigned long long* ws = static_cast<unsigned long long*>(fs.soft_ws);
    if (soft) fast_init_soft_kernel<<<(unsigned)((pairs + 255) / 256), 256, 0, stream>>>(ws, pairs, pd.counters);
    else fast_init_kernel<<<(unsigned)((pairs + 255) / 256), 256, 0, stream>>>(feat_i, pairs, pd.counters);
    count_launch();
    // the batch goes through in chunks of a few examples: the shifted copies of a chunk are read while
    // they are still in L2, and they stay small
    const int n_chunks = (int)(((int64_t)N + chunk - 1) / chunk);
    if (fs.profile) {
        while ((int)fs.evs.size() < 3 * n_chunks) {
            cudaEvent_t ev = nullptr;
            if ((e = cudaEventCreate(&ev)) != cudaSuccess) return e;
            fs.evs.push_back(ev);
        }
        fs.ev_chunks = 0;
    }
    for (int c = 0; c < n_chunks; ++c) {
        const int n0 = c * chunk, nc = std::min(chunk, N - n0);
        if (X_u8) {   // the kernels read the normalised samples from the unshifted zero-margined copy
            a.X = streamed ? fs.wpad + fs.host.wfront : fs.xpad + kTPadFront;
            a.x_row_stride = streamed ? kWCopies * fs.host.wpitch : fs.host.pad_pitch;
        } else {
            a.X = X + (size_t)n0 * dp.C * dp.L;
            a.x_row_stride = dp.L;
        }
        a.feat_i = feat_i + (size_t)n0 * 2 * dp.K;
        a.ws = ws ? ws + (size_t)n0 * 2 * dp.K : nullptr;
        a.N = nc;
        if (c > 0) {
            e = cudaMemsetAsync(pd.counters, 0, 8, stream);
            if (e != cudaSuccess) return e;
        }
        if (X_u8 && streamed) {
            stream_copy_u8_kernel<<<sms * 8, 256, 0, stream>>>(X_u8 + (size_t)n0 * dp.C * dp.L, fs.wpad, (int64_t)nc * dp.C, dp.L, dp.C,
                                                               fs.host.wpitch, (int)fs.host.wfront, *norm);
            count_launch();
        } else if (streamed) {
            launch_stream_copy(fs, a.X, (int64_t)nc * dp.C, dp.L, sms, c == 0, stream);
        } else if (X_u8) {
            fast_pad_copy_u8_kernel<<<sms * 8, 256, 0, stream>>>(
                reinterpret_cast<const uchar4*>(X_u8 + (size_t)n0 * dp.C * dp.L), fs.xpad, (int64_t)nc * dp.C, dp.L / 4, dp.C,
                fs.host.pad_pitch, kTPadFront, fs.copy_floats, *norm);
            count_launch();
        } else if (pd.n_titems > 0) {
            launch_pad_copy(fs, a.X, (int64_t)nc * dp.C, dp.L, sms, stream);
        }
        if (fs.profile) cudaEventRecord(fs.evs[3 * c], stream);
        if (pd.n_sitems > 0) launch_s(a, fs, soft ? 1 : half ? 3 : 0, sms, c == 0 || streamed || copied, stream);
        if (fs.profile) cudaEventRecord(fs.evs[3 * c + 1], stream);
        if (streamed) {
            launch_stream(a, soft ? 1 : half ? 3 : 0, sms, l2, pd.n_sitems > 0, stream);
        } else if (pd.n_titems > 0) {
            const unsigned grid = t_grid(nc, pd.n_titems, sms);
            if (soft) fast_t_forward<1><<<grid, kTBlockThreads, t_bytes, stream>>>(a);
            else if (half) fast_t_forward<3><<<grid, kTBlockThreads, t_bytes, stream>>>(a);
            else fast_t_forward<0><<<grid, kTBlockThreads, t_bytes, stream>>>(a);
            count_launch();
        }
        if (fs.profile) {
            cudaEventRecord(fs.evs[3 * c + 2], stream);
            fs.ev_chunks = c + 1;
        }
    }
    const int64_t fin = (int64_t)N * pd.n_krec;
    if (fin > 0) {
        // in stream order: behind the stream kernel alone it would not wait for the small-dilation kernel
        if (soft) fast_finalize_soft_kernel<<<(unsigned)((fin + 255) / 256), 256, 0, stream>>>(feat, argmax, ws, pd.krec, pd.n_krec, N, dp.K);
        else fast_finalize_kernel<<<(unsigned)((fin + 255) / 256), 256, 0, stream>>>(feat, pd.krec, pd.n_krec, N, dp.K);
        count_launch();
    }
    return cudaGetLastError();
}

cudaError_t launch_fast_backward(FastState& fs, const DeviceParams& dp, int64_t n_weights, const float* X, int N,
                                 float lambda, float shift, const float* dfeat, const int32_t* argmax, float* dW,
                                 float* db, cudaStream_t stream) {
    std::lock_guard<std::mutex> lk(fs.mu);
    const int sms = fs.sms, l2 = fs.l2_bytes;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = set_kernel_attributes(dev, fs.host);
    if (e != cudaSuccess) return e;
    const size_t t_bytes = t_smem_bytes();
    const PlanDevice& pd = fs.dev;
    // workspace: fixed-point sums [n_weights + K], scales [K], max |x| (fixed size per handle)
    const size_t acc_bytes = align256((size_t)(n_weights + dp.K) * 8), scale_bytes = align256((size_t)dp.K * 8);
    if ((e = ensure_bwd_ws(fs, dp, n_weights)) != cudaSuccess) return e;
    long long* accfix = static_cast<long long*>(fs.bwd_ws);
    double* scale = reinterpret_cast<double*>(static_cast<char*>(fs.bwd_ws) + acc_bytes);
    unsigned* absmax = reinterpret_cast<unsigned*>(static_cast<char*>(fs.bwd_ws) + acc_bytes + scale_bytes);
    const bool streamed = pd.n_wunits > 0, copied = pd.n_titems > 0;
    int chunk = chunk_examples(fs, dp.C, streamed, copied);
    const bool resident = resident_backward(fs.host);
    if (N > 0 && !resident) {
        if (streamed) e = ensure_stream_capacity(fs, std::min(N, chunk), dp.C, dp.L);
        else if (copied) e = ensure_pad_capacity(fs, std::min(N, chunk), dp.C, dp.L);
        if (e != cudaSuccess) return e;
        if (streamed || copied) chunk = std::min(chunk, fs.most_examples);
    }
    const int64_t n_x = (int64_t)N * dp.C * dp.L;
    const bool small = n_x > 0 && n_x <= kSmallBatch;
    if (!small && (e = cudaMemsetAsync(absmax, 0, 256, stream)) != cudaSuccess) return e;
    if (n_x > 0 && !small) {
        auto blocks = [&](int64_t loads) { return (unsigned)std::min<int64_t>(sms * 8, (loads + 1023) / 1024); };   // four loads per thread
        if (dp.L % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0)
            fast_absmax_kernel<<<blocks(n_x / 4), 256, 0, stream>>>(reinterpret_cast<const float4*>(X), n_x / 4, absmax);
        else fast_absmax_scalar_kernel<<<blocks(n_x), 256, 0, stream>>>(X, n_x, absmax);
        count_launch();
    }
    const float* none = nullptr;
    if (n_x > 0 && !small)
        launch_dependent(fast_bwd_prepare_kernel, (pd.n_krec + 7) / 8, 256, 0, stream, dfeat, pd.krec, pd.n_krec, N, dp.K, lambda, absmax, none, 0, scale,
                         accfix, n_weights, pd.counters);
    else
        fast_bwd_prepare_kernel<<<(pd.n_krec + 7) / 8, 256, 0, stream>>>(dfeat, pd.krec, pd.n_krec, N, dp.K, lambda, absmax, small ? X : none,
                                                                         (int)(small ? n_x : 0), scale, accfix, n_weights, pd.counters);
    count_launch();
    FwdArgs a;
    a.plan = fs.dev; a.feat_i = nullptr; a.ws = nullptr;
    a.c1 = lambda * 1.4426950408889634f; a.c0 = -shift * 1.4426950408889634f;
    a.C = dp.C; a.L = dp.L; a.K = dp.K;
    a.accfix = accfix; a.scale = scale; a.n_weights = n_weights; a.lambda = lambda;
    a.x_row_stride = dp.L;
    if (resident && N > 0) {
        ResidentArgs r = resident_args(fs, dp, X, N, lambda, shift);
        r.dfeat = dfeat; r.argmax_in = argmax; r.accfix = accfix; r.scale = scale; r.n_weights = n_weights;
        launch_resident(r, fs.host, 2, sms, stream);
    }
    for (int n0 = 0; n0 < N && !resident; n0 += std::min(chunk, N - n0)) {
        const int nc = std::min(chunk, N - n0);
        a.X = X + (size_t)n0 * dp.C * dp.L;
        a.dfeat = dfeat + (size_t)n0 * 2 * dp.K;
        a.argmax = argmax + (size_t)n0 * dp.K;
        a.N = nc;
        if (n0 > 0 && (e = cudaMemsetAsync(pd.counters, 0, 8, stream)) != cudaSuccess) return e;
        if (streamed) launch_stream_copy(fs, a.X, (int64_t)nc * dp.C, dp.L, sms, n0 == 0, stream);
        else if (copied) launch_pad_copy(fs, a.X, (int64_t)nc * dp.C, dp.L, sms, stream);
        if (pd.n_sitems > 0) launch_s(a, fs, 2, sms, n0 == 0 || streamed || copied, stream);
        if (streamed) {
            launch_stream(a, 2, sms, l2, pd.n_sitems > 0, stream);
        } else if (pd.n_titems > 0) {
            fast_t_forward<2><<<t_grid(nc, pd.n_titems, sms), kTBlockThreads, t_bytes, stream>>>(a);
            count_launch();
        }
    }
    fast_bwd_finalize_kernel<<<(pd.n_krec + 7) / 8, 256, 0, stream>>>(accfix, scale, pd.krec, pd.n_krec, n_weights, dW, db);
    count_launch();
    return cudaGetLastError();
}

}  // namespace fast
}  // namespace rocket
