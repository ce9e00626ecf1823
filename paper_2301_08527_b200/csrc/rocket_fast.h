// Fast path of the forward transform: data structures shared by the host planner and the
// fused kernels.
//
// Geometry.  A kernel with dilation d reads x[u + j*d] for output u = i - p (i the output
// index, p the padding).  Writing u = t*d + r with 0 <= r < d turns the series into a 2-D array
// A[t][r] = x[t*d + r], and the dilated convolution into a dense length-len filter down the
// columns of A: output (t, r) needs A[t .. t+len-1][r].  A thread owns two adjacent columns
// and 16 consecutive rows, keeps the 32 accumulators in registers as 16 packed pairs and
// streams 16+len-1 input pairs per channel past them with packed two-wide FMAs
// (fma.rn.f32x2), so every input is loaded once and used len times.  Lanes of a warp own
// adjacent column pairs: a warp tile is 16 rows x 64 columns.
//
// Three kernels share the arithmetic core:
//   S (d < split): kernels of one dilation form a bucket.  Columns of successive bands of kRS rows
//     are strung together into one "raster" (band-major, r-minor) and a tile is 64 consecutive
//     raster positions, so lanes stay busy even when d < 64.  A block stages one tile of ALL
//     channels in shared memory, then its warps pull kernels of the bucket from a shared
//     counter, so one staged tile serves dozens to hundreds of kernels.
//   stream (d >= split; rocket_stream.cu): few kernels share a dilation, so every warp takes tiles of
//     one kernel of its own and streams the kernel's channels through its own shared memory.
//   T (d >= split, handles with dilations near L / 3.5 and above, for which the stream kernel's copies
//     would be mostly margins): a block of eight consumer warps takes one
//     kernel and one tile of up to eight warp tiles (128 x 64, 64 x 128, 32 x 256, or 16 x 512 for
//     kernels whose outputs span at most 16 rows of A) and streams the kernel's channels through a
//     ring of shared-memory stages.  A producer warp fills the
//     ring with tiled TMA loads from a zero-margined copy of the batch, viewed as a 3-D tensor
//     (x within a run of 4d floats, y = which run, z = channel row): rows s, s+4, s+8, .. of
//     a tile are then one box, and four boxes (one per s mod 4) bring a whole stage without
//     spending issue slots of the consumer warps.
#pragma once

#include <cstdint>
#include <mutex>
#include <vector>

#include "rocket_internal.h"

#ifdef __CUDACC__
#define ROCKET_CX __host__ __device__ constexpr
#else
#define ROCKET_CX constexpr
#endif

namespace rocket {
namespace fast {

constexpr int kR = 16;                                             // output rows of a warp tile
constexpr int kWarpCols = 64;                                      // columns of a warp tile (2 per lane)
constexpr int kRowsMax = kR + ROCKET_MAX_LENGTH - 1;               // staged rows a warp tile reads
#ifndef ROCKET_SPLIT
#define ROCKET_SPLIT 64
#endif
// S below, stream (or T) at or above.  The stream kernel's tiles are 64 columns of one band, so it cannot start lower; with 96 to
// 256 the S kernel's buckets hold too few kernels for the 16 warps of a block (the hard transform loses 0.5 to 4 %).
constexpr int kSplitDefault = ROCKET_SPLIT;
constexpr int kTMinDilation = 64;                                  // a T tile needs 64 residues in one band

// ---- kernel record: one fast kernel as the device reads it (header + duplicated weights) ----
constexpr int kPairRow = 24;                                       // floats of one channel's weight row
struct alignas(16) KRec {
    int32_t len, d, p, m;
    int32_t nout, k, lo_u, hi_u;   // k: original kernel index; lo_u = -p; hi_u = nout - p (exclusive)
    float negb;                    // 0 - bias (never -0.0)
    int32_t ch[ROCKET_MAX_CHANNELS_PER_KERNEL];   // S regime: positions in the bucket's channel list
    int32_t tl, rl, th, rh;        // lo_u = tl * d + rl and hi_u = th * d + rh with 0 <= rl, rh < d
    int32_t woff;                  // offset of the kernel's weights in the caller's ragged weight array
    int32_t pad_[7];
    // w2[q][2j] = w2[q][2j+1] = 0 - W[q][j]: each weight twice, ready as a packed pair
    float w2[ROCKET_MAX_CHANNELS_PER_KERNEL][kPairRow];
};
static_assert(sizeof(KRec) == 128 + 4 * ROCKET_MAX_CHANNELS_PER_KERNEL * kPairRow, "KRec layout");
static_assert(sizeof(KRec) % 16 == 0, "KRec must be copyable in 16-byte pieces");

// ---- S regime --------------------------------------------------------------------------------
// Per-channel feature scaling of 8-bit input (Section 4.3): x = (v - mean[c]) * inv_std[c].
constexpr int kNormMaxChannels = 20;
struct NormArgs { float mean[kNormMaxChannels], inv_std[kNormMaxChannels]; };

constexpr int kSMaxPlanes = 20;                                    // (example, channel) planes the S tile can stage
constexpr int kF16MaxChannels = 20;                                // what rocket_transform_f16 is documented to take
constexpr int kMaxChannels = 255;                                  // channels of a series the fused kernels take (stored as bytes)
// Output rows of a warp tile in the S regime (the band height of its rasters).  More rows per thread than in
// the T regime: the work per (kernel, tile) grows while the per-kernel bookkeeping and the rows staged per
// output shrink.  Measured at 60 x 20 x 50,000 (hard): 16 rows 25.7 ms, 20 rows 24.9, 22 rows 24.6, 24 to 26
// rows 24.1 (16 warps each; 12 warps are slower at every height), 28 rows need 14 warps for the tile to fit.
#ifndef ROCKET_S_ROWS
#define ROCKET_S_ROWS 24
#endif
#ifndef ROCKET_S_THREADS
#define ROCKET_S_THREADS 512
#endif
constexpr int kRS = ROCKET_S_ROWS;
static_assert(kRS >= 8 && kRS <= 32, "the row masks of the pooling hold at most 32 rows");
constexpr int kSRowsMax = kRS + ROCKET_MAX_LENGTH - 1;             // staged rows an S warp tile reads
// Handles whose columns fill their last tiles badly at that height take a lower one (the planner's estimate decides; wide handles don't).
constexpr int kSLowRows[2] = {21, 18};
constexpr int kSThreads = ROCKET_S_THREADS, kSWarps = kSThreads / 32;   // one block per SM
constexpr int kSPlaneFloats = kSRowsMax * kWarpCols;               // one channel of an S tile
// Wide handles: the kernels of some dilation use more than kSMaxPlanes channels, none more than kSWidePlanes.  Their tiles are staged in two halves of kRS / 2
// rows, of which kSWidePlanes planes fit, so that a dilation stays one bucket.  With buckets of 20 channels the
// 200 kernels of a dilation over 32 channels were 15 buckets of a dozen kernels each, and a tile's copies took longer than the
// work on it (24 x 32 x 1,751, 2,000 kernels).
constexpr int kSHalfRows = kRS / 2, kSWidePlanes = 34;
ROCKET_CX int s_plane_floats(int rows) { return (rows + ROCKET_MAX_LENGTH - 1) * kWarpCols; }
constexpr int kSManyKernels = 32, kSSomeKernels = 8;               // buckets below these share a tile among several examples
constexpr int kSLengthOrderMin = 100;                              // buckets from this many kernels up are ordered by length

// The kernels of a bucket use at most kSMaxPlanes channels between them (kSWidePlanes in a wide handle): where the kernels of one
// dilation use more, they are several buckets.  Their records hold positions in the bucket's channel list.
struct SBucket {
    int32_t d, tmin, nbands, raster_len;  // raster_len = nbands * d
    int32_t kbeg, kend, rows, nch;        // kernels [kbeg, kend) of krec; rows = s_rows + max len - 1; channels used
    uint8_t ch[40];                       // the channels (at most kSWidePlanes)
    int32_t pad_[2];
};
constexpr int kSBucketWords = 20;
static_assert(sizeof(SBucket) == 4 * kSBucketWords && kSWidePlanes <= 40, "SBucket layout");
// One S tile: 64 raster positions from c0 of a bucket.  interior = 1 when every (row, column) of the
// tile is an output of every kernel of the bucket (then the kernels need no range tests).
struct SItem { int32_t bucket, c0, interior, pad_; };

// ---- T regime --------------------------------------------------------------------------------
// Consumer warps per block, blocks per SM and ring depth of the T kernel.  A block's consumer warps move
// through a stage in step, so the number of independent blocks per SM decides how often the FMA pipes
// find a warp that is ready.
#ifndef ROCKET_T_WARPS
#define ROCKET_T_WARPS 8
#endif
#ifndef ROCKET_T_BLOCKS
#define ROCKET_T_BLOCKS 2
#endif
#ifndef ROCKET_T_STAGES
#define ROCKET_T_STAGES 2
#endif
constexpr int kTConsumerWarps = ROCKET_T_WARPS;
static_assert(kTConsumerWarps == 4 || kTConsumerWarps == 8, "tile shapes are laid out for 4 or 8 consumer warps");
constexpr int kTBlocksPerSM = ROCKET_T_BLOCKS;
constexpr int kTThreads = 32 * (kTConsumerWarps + 1);              // one group: consumer warps + one producer warp
// Groups per block: every group is a producer with its consumers, its own ring and its own stream of tiles.
// Two groups in one block instead of two blocks of one group leave more registers to every thread (the
// register file is handed out per pair of warps, and a group has an odd number of warps).
#ifndef ROCKET_T_GROUPS
#define ROCKET_T_GROUPS 1
#endif
constexpr int kTGroups = ROCKET_T_GROUPS;
constexpr int kTBlockThreads = kTGroups * kTThreads;
constexpr int kTStages = ROCKET_T_STAGES;
constexpr int kTParamSlots = kTStages + 2;
// A T tile is rg row groups x cg column groups of warp tiles, rg * cg <= the consumer warps, cg in {1, 2, 4}
// (cg = 4 only with 8 consumer warps: a 16 x 256 tile would load 26 rows for 16 rows of outputs).
// One box per phase brings all column groups (64 * cg floats wide).  The zero-margined copy is kept
// four times, shifted by 0, 1, 2 and 3 floats, so that every row start is 16-byte aligned in one
// of them: a box needs no alignment slack and every pair a consumer reads is 8-byte aligned.
constexpr int kTMaxCg = kTConsumerWarps >= 8 ? 4 : 2;
ROCKET_CX int t_box_cols(int cg) { return kWarpCols * cg; }
// Box rows of one phase (rows s, s+4, ..), and the floats of one phase box (a multiple of 64
// floats, so every box destination stays 128-byte aligned).
ROCKET_CX int t_box_rows(int rg, int len) { return (kR * rg + len - 1 + 3) / 4; }
ROCKET_CX int t_phase_floats(int cg, int box_rows) { return box_rows * t_box_cols(cg); }
ROCKET_CX int t_stage_floats(int rg, int cg, int len) { return 4 * t_phase_floats(cg, t_box_rows(rg, len)); }
ROCKET_CX int imax_cx(int a, int b) { return a > b ? a : b; }
constexpr int kTStageFloats =
    imax_cx(imax_cx(t_stage_floats(kTConsumerWarps, 1, ROCKET_MAX_LENGTH), t_stage_floats(kTConsumerWarps / 2, 2, ROCKET_MAX_LENGTH)),
            kTMaxCg >= 4 ? t_stage_floats(kTConsumerWarps / 4, 4, ROCKET_MAX_LENGTH) : 0);
constexpr int kTChunkTiles = 4;                                    // consecutive tiles a block draws at a time
constexpr int kTWideCols = 256;                                    // columns of one half of a wide tile
constexpr int kTWideHalves = kTConsumerWarps / 4;                  // a wide tile is one row of all consumer warps' tiles
constexpr int kChunkExamples = 12;                                // examples per pass through the fused kernels, at least
constexpr int kTPadFront = 128;                                    // zero floats before every channel row
constexpr int kTXExtra = 256;                                      // floats a box may run past a 4d run

// One T tile with everything the producer warp needs (32 words).
struct alignas(16) TItem {
    int32_t map, t0, r0, rg;              // map: index of the tile's tensor map; tile origin (t0, r0)
    int32_t d, len, m, box_rows;
    uint8_t ch[12];
    int32_t krec;                         // index into the kernel records
    int32_t cg, wide, g_lo, g_hi;         // wide tile: one row of warp tiles in halves of 256 columns, of which only
                                          // the groups of four rows [g_lo, g_hi) are loaded (box_rows = g_hi - g_lo)
    int32_t x[4], y[4];                   // tensor coordinates of the four phase boxes (first half; y of group g_lo)
    int32_t j[4];                         // which shifted copy each phase reads
    // bit w: every output of consumer warp w's warp tile exists (no range tests needed) / at least one does
    int32_t warp_interior, warp_active;
    int32_t pad1_[2];
};
static_assert(sizeof(TItem) == 128, "TItem must be 32 words");
// ---- stream regime (rocket_stream.cu): the large dilations, one warp per tile ------------------
constexpr int kWRows = 16;                                         // highest band
constexpr int kWWarps = 16, kWThreads = 32 * kWWarps;              // independent warps of the one block per SM
constexpr int kWStages = 2;                                        // (tile, channel) visits in flight per warp
constexpr int kWStageFloats = (kWRows + ROCKET_MAX_LENGTH - 1 + 3) / 4 * 4 * kWarpCols;   // input rows of a visit, whole y steps
constexpr int kWCopies = 7;                                        // shifted copies of every channel row, next to one another
constexpr int kWUnitVisits = 16, kWItemVisits = 32;                // visits of a unit, and of a unit for a group of examples
constexpr int kWSoftSetItems = 24;                                 // items per warp of a set, soft and backward
// What the copies of a pass take: 800 MB (13 examples of 20 x 50,000), or four examples where those take no more than 4 GB.
constexpr int64_t kWCopyBytes = 800ll << 20, kWMostCopyBytes = 4ll << 30;
constexpr int kWFewExamples = 4;

// A unit of work: consecutive tiles of one kernel (32 words).  The kernel's output rows from t0 on are cut into bands of R rows,
// a band into ncol tiles of 64 columns; tile number band * ncol + column group.
struct alignas(16) WUnit {
    int32_t krec, map, t0, tile0;         // tile0: the unit's first tile
    int32_t ntiles, shape, d, m;          // shape: R | len << 8 | row_xor << 16 (stage row of input row s: s ^ row_xor in its four)
    int32_t k, lo_u, hi_u, p;
    int32_t tl, rl, th, rh;
    int32_t nout, woff, ncol, band_y;     // band_y: y steps from band to band
    int32_t x0, y0, run, copy;            // coordinates of the first column of band 0; floats per y step; first copy
    uint8_t ch[12];
    int32_t bytes, span, pad_[3];         // bytes of a visit's copy; positions from a band's first row to its last (w_span)
};
static_assert(sizeof(WUnit) == 128, "WUnit must be 32 words");
// Examples of a pass of the stream regime for rows of `pitch` floats.
int stream_chunk(int C, int64_t pitch);
// Capacity for `want` examples, or as many as there is room for: alloc(n) makes room for n examples.  0 when there is none for one.
template <class Alloc>
int fit_examples(int want, Alloc&& alloc) {
    for (int n = want; n >= 1; n /= 2)
        if (alloc(n)) return n;
    return 0;
}
// How a pass of N examples is handed out to the warps of the stream kernel (mode: 0 = hard, 1 = soft, 2 = backward, 3 = hard in half
// precision): an item is a unit for `examples` examples, the items of `groups_per_set` such groups go through all units together.
struct StreamItems { int examples, groups, groups_per_set; };
StreamItems stream_items(int N, int C, int L, int n_units, double visits, int mode, int sms, int64_t l2_bytes);
// One tensor map of the stream regime: boxes of 64 columns x y_rows y steps over the copies, for dilation d.
struct WMapSpec { int32_t d, y_rows; };
// Rows per y step: an odd dilation takes four rows (one per alignment) as a dimension of their own, d = 2 mod 4 two.
ROCKET_CX int w_rows_per_y(int d) { return d % 4 == 0 ? 1 : d % 4 == 2 ? 2 : 4; }

// One tensor map: boxes of box_cols x box_rows floats over runs of 4 * d floats.
struct TMapSpec { int32_t d, box_cols, box_rows; };

// ---- resident regime (rocket_resident.cu): short series, whole examples in shared memory ------
// Heights of its bands.  Odd: neighbouring columns of a band row lie side by side and those of the next band an odd number of rows further on, so
// that a warp's loads meet few times in a shared-memory bank, at dilation 1 too, where 16 rows would meet sixteen times.  A tile is 64
// columns, so that what decides is how many tiles a series fills.
// Forward: 17 and 11 rows (bands = 0), 9 and 5 (1) where series are too short for those 64 columns, 21 and 11 (2) just beyond what one tile of
// 17 rows holds.  Hard, us: 100 x 1 x 64 and 5,000 kernels 329 with 17 and 11 rows, 289 with 15 and 9; 120 x 1 x 1,180 and 10,000 kernels 1,626
// with 17 and 11, 1,379 with 21 and 11 (20 warps; 18: 1,414).
// Backward: one height, 5, 7, 9 or 11 (3 to 6).  It runs a convolution and a gradient per length and height, more code than the instruction
// caches hold (at 17 and 11 rows 40 % of the issue slots were used, with more than half of a warp's stalls for instructions): less code
// is worth more than the reads that higher bands save.  24 x 6 x 900 and 2,000 kernels 312 us before, 360 at 17 and 11 rows, 233 at 9; 100 x 6 x
// 640 and 5,000 kernels 2,480, 1,915, 1,475 (11; 13: 1,970); 100 x 6 x 1,900 and 5,000 4,560, 3,840 (tile kernels), 3,647; 100 x 6 x 200 and
// 5,000 2,527, 905 (9 and 5 rows, 16 warps), 812 (5 rows).
ROCKET_CX int resident_high(int bands) { return bands >= 3 ? 2 * bands - 1 : bands == 2 ? 21 : bands == 1 ? 9 : 17; }
ROCKET_CX int resident_low(int bands) { return bands >= 3 ? 2 * bands - 1 : bands == 1 ? 5 : 11; }
constexpr int kRBackBands[4] = {3, 4, 5, 6};
// Warps of a block (mode: 0 = hard, 1 = soft, 2 = backward, 3 = hard in half precision).
ROCKET_CX int resident_warps(int mode, int bands) { return mode == 2 || mode == 1 || bands == 2 ? 20 : bands == 1 ? 28 : 24; }
constexpr int kRMostFloats = 57600;                                // what shared memory holds: examples, rows padded to 16 bytes
// The longest series: beyond, a pair is a warp's for too long where there are few, and the other kernels' larger tiles are as good where there
// are many (us, before and with this kernel: 1 x 3 x 5,000, 10,000 kernels 192 and 97, 100 x 3 x 5,000, 5,000 kernels 2,825 and 2,842; 8 x 3 x
// 18,000, 1,000 kernels 205 and 257).  The second where tiles test their reads (24 x 32 x 1,751, 2,000 kernels 477 and 218; 8 x 9 x 6,000,
// 1,000 kernels 142 and 240).
constexpr int kRMostSteps = 5000, kRMostStepsTested = 2048;
constexpr int kRSmallSteps = 1024, kRTallSteps = 1600;             // steps up to which the low bands are considered, and from there the tallest
constexpr int kRMostOutputs = 1 << 20;                             // outputs and dilation up to which columns are counted exactly in FP32

// One kernel (32 words).  Its outputs, counted from the first one, are t d + r for t < nq + (r < nr); the input rows of column r that
// are samples, or zeros next to them in shared memory, are t from pq + (r < pr) to lq + (r < lr), exclusive.
struct alignas(16) RUnit {
    int32_t krec, k, len, d;
    int32_t m, nout, p, high;             // high, low: bands of the greater height, then bands of the lesser
    int32_t low, nq, nr, pq;
    int32_t pr, lq, lr;
    float inv_d;
    uint8_t ch[12];
    int32_t woff, pad_[12];
};
static_assert(sizeof(RUnit) == 128, "RUnit must be 32 words");
// How a call of N examples is dealt to the blocks: tasks of `examples` examples and every parts-th kernel, of which a warp takes one for
// `run` of the examples at a time, or for one of them every split-th tile.
struct ResidentSplit { int examples, groups, parts, run, split; unsigned grid; };

struct PlanHost {
    bool enabled = false;
    bool resident = false;                // the examples fit the resident kernel's shared memory
    int r_bands = 0, r_back = 0;          // the heights of its bands; those of the backward's, 0 if it does not serve it
    bool r_zeros = false;                 // and so do zeros around every row, as far as any tile reads
    std::vector<RUnit> runits;
    int r_front = 0, r_pitch = 0;         // floats of zeros in front of the first channel row in shared memory; from row to row
    int r_tiles = 0;                      // most tiles of a kernel
    double r_clocks = 0.0, r_longest = 0.0;   // resident kernel: clocks of an SM for one example, and of a warp for its longest pair
    int r_tiles_from = 0;                 // examples from which a hard transform goes to the tile kernels all the same; 0: never
    int split = kSplitDefault;
    std::vector<KRec> krec;
    std::vector<SBucket> sb;
    std::vector<SItem> sitems;
    std::vector<TItem> titems;            // kernel by kernel, in the order the blocks walk them
    std::vector<TMapSpec> tmaps;          // tensor maps the T tiles refer to
    std::vector<WUnit> wunits;            // stream regime; empty when its copies would need too much room
    std::vector<WMapSpec> wmaps;
    double w_visits = 0.0;                // (tile, channel) visits of one example
    int64_t wfront = 0, wpitch = 0;       // zeros before the first channel row; floats from copy to copy
    std::vector<int32_t> generic_list;    // kernels the fast path does not take
    int64_t pad_pitch = 0;                // floats per channel row of the zero-margined copy
    int s_max_nch = 0;                    // most channels of any S bucket
    bool s_wide = false;                  // the S tiles are staged in halves of up to kSWidePlanes planes
    int s_rows = kRS;                     // rows of a band of the S tiles
    int s_class_end[3] = {0, 0, 0};       // S tiles by kernels in their bucket: at least kSManyKernels, kSSomeKernels, fewer
    double flops_s = 0.0, flops_t = 0.0;  // conv flop of one example in either regime
    // What generic_pays compares, in us: work of one example for one SM (small dilations) and for the GPU (large dilations and their
    // copies, generic kernels), and what one tile or one kernel takes at least.
    double us_s = 0.0, us_s_tile = 0.0, us_t = 0.0, us_g = 0.0, us_g_kernel = 0.0;
};

// Whether the generic kernels serve a call of N examples in less time than the fused ones (asked where C > kSMaxPlanes); soft: the
// soft transform or its backward.
bool generic_pays(const PlanHost& plan, int N, int sms, bool soft);
// A bound on the examples of the calls of up to max_N that the generic kernels serve for that reason (pays), or that the fused ones do:
// what either needs a workspace for.
int pays_up_to(const PlanHost& plan, int max_N, int sms, bool soft, bool generic);

// How the S kernel's tiles are shared among the examples of a pass: tiles [end[i - 1], end[i]) for examples[i] examples together, as
// groups[i] groups; grid: its blocks.
struct SGroups { int end[3], examples[3], groups[3]; unsigned grid; };
SGroups s_groups(const PlanHost& plan, int N, int sms);

ResidentSplit resident_split(const PlanHost& plan, int N, int C, int sms, int mode);
// And for the pairs of a task whose tiles several warps share (all modes but the backward, which adds up in global memory anyway).
constexpr int kRMergeFloats = 8;
inline int64_t resident_merge_floats(const PlanHost& plan, int64_t n, int parts, int split, int mode) {
    return split > 1 && mode != 2 ? kRMergeFloats * n * ((int64_t)plan.runits.size() / parts + 1) : 0;
}
// The backward, whose code is twice as long and whose sums leave the warp once per tile, only where no tile has to test its reads: handles with room
// for the zeros of its height (us, before and with this kernel, 2,000 kernels: 100 x 6 x 1,251 1,307 and 1,124, 60 x 3 x 5,000 1,850 and 1,615).
inline bool resident_backward(const PlanHost& plan) { return plan.r_back != 0; }
// Whether every fused call of the handle is a matter of one kernel, or of tiles of at most kSMaxPlanes channels: no call of such a handle is
// better served by the generic kernels, and generic_pays is not asked.
inline bool always_fused(const PlanHost& plan, int C, bool backward) {
    return C <= kSMaxPlanes || (backward ? resident_backward(plan) : plan.resident);
}
// Hard transforms of many kernels on many examples, from 1,345 steps on: copying a tile per dilation is then spread over hundreds of kernels,
// and the tile kernels' inner loops, whose addresses are constants, are the faster ones.  Measured (us, tile kernels and resident, 20,000
// kernels): 100 x 6 x 1,400 4,738 and 5,100, 100 x 20 x 1,400 5,984 and 6,374, 100 x 6 x 2,300 6,925 and 7,821; on the other side of the lines
// 24 x 6 x 1,400 1,390 and 1,230, 60 x 6 x 1,400 and 3,000 kernels 528 and 506, 128 x 3 x 1,560 2.5 % and 60 x 1 x 1,700 and 10,000 11 % in the
// resident kernel's favour.  One size behind them is slower, 60 x 2 x 3,200 and 10,000 kernels by 2 %.  The soft modes and half precision are
// faster with the resident kernel throughout.  Handles of such sizes hold both plans (20,000 kernels: created in 48 ms where 32 do).
constexpr int kRTilesSteps = 1345, kRTilesMidSteps = 1500, kRTilesFarSteps = 2048, kRTilesKernels = 10000;
constexpr double kRTilesPairs = 1.2e6, kRTilesFarPairs = 6e5;      // (kernel, example) pairs; beyond kRTilesFarSteps steps
inline bool resident_forward(const PlanHost& plan, int N, bool hard) { return plan.resident && !(hard && plan.r_tiles_from > 0 && N >= plan.r_tiles_from); }
// Floats of shared memory for n examples.
inline int64_t resident_floats(const PlanHost& plan, int64_t n, int C) { return plan.r_front + n * C * plan.r_pitch; }

struct PlanDevice {
    const KRec* krec = nullptr;
    const RUnit* runits = nullptr;
    const SBucket* sb = nullptr;
    const SItem* sitems = nullptr;
    const TItem* titems = nullptr;
    const WUnit* wunits = nullptr;
    const void* wmaps = nullptr;          // CUtensorMap[n_wmaps]
    const int32_t* generic_list = nullptr;
    unsigned* counters = nullptr;         // [0] S work counter, [1] T work counter
    int* error_flag = nullptr;            // set when a bounded wait gave up
    const void* tmaps = nullptr;          // CUtensorMap[n_tmaps], 128 bytes each
    float* xpad = nullptr;                // zero-margined copy of the batch
    int64_t pad_pitch = 0;
    int n_krec = 0, n_sitems = 0, n_titems = 0, n_generic = 0, n_tmaps = 0, n_wunits = 0;
    double w_visits = 0.0;                // (tile, channel) visits of one example in the stream kernel
};

// Writes kernel f.k's bias and weights (negated, every weight twice) into its record.
void fill_record_weights(const HostParams& hp, KRec& f);
// Copies the records of the host plan to the device again (after their weights changed).
cudaError_t upload_records(FastState& fs);

// Builds the launch plan for the kernels in hp (host side, once per handle).  all_tiles: also the T tiles of kernels that have
// stream units, which no launch uses, and S bands of kRS rows.  only_used: no tiles and units at all where the resident kernel serves every
// pass of the handle.
void build_plan(const HostParams& hp, int split, PlanHost& out, bool all_tiles = true, bool only_used = false);

// Device-side state of the fast path owned by a handle.
struct FastState {
    std::mutex mu;                        // guards the grow-only buffers below and the launch sequence of a call
    int sms = 0, l2_bytes = 0;            // of the handle's device
    PlanHost host;
    PlanDevice dev;
    void* plan_blob = nullptr;            // records, buckets, items, counters, error flag
    void* maps_blob = nullptr;            // tensor maps
    float* xpad = nullptr;                // the four shifted zero-margined copies, capacity pad_examples
    int pad_examples = 0;
    int most_examples = 1 << 30;          // of either kind of copies: fewer than wanted once there was no room for more (until the next reserve)
    int64_t copy_floats = 0;              // floats of one copy
    float* wpad = nullptr;                // stream regime: the seven shifted copies, capacity wpad_examples
    int wpad_examples = 0;
    void* wmaps_blob = nullptr;
    void* soft_ws = nullptr;              // soft mode: 16 bytes per (example, kernel), grows with N
    size_t soft_ws_bytes = 0;
    void* bwd_ws = nullptr;               // backward: fixed-point sums [n_weights + K], scales [K], max |x|
    bool profile = false;                 // record events around the S and T launches
    std::vector<cudaEvent_t> evs;         // three per chunk: before S, between S and T, after T
    int ev_chunks = 0;                    // chunks of the last profiled call
};

// Uploads the plan (once per handle, at binding).
cudaError_t upload_plan(FastState& fs);
// Frees everything upload_plan / ensure_pad_capacity allocated.
void release_fast_state(FastState& fs);
// The same for the stream regime's copies.
cudaError_t ensure_stream_capacity(FastState& fs, int N, int C, int L);
// Makes the padded copy hold N examples, or as many as there is room for (at least one, or cudaErrorMemoryAllocation), and
// (re-)encodes the tensor maps over it.
cudaError_t ensure_pad_capacity(FastState& fs, int N, int C, int L, bool without_maps = false);

// Allocates, once, everything the fused kernels need for calls of up to max_N examples (the zero-margined
// copies and their tensor maps, the soft transform's and the backward's workspaces) and opts the kernels
// into their shared-memory sizes; later calls within that size allocate nothing.
// again: the full size, where there was no room for it before.
cudaError_t reserve_fast_state(FastState& fs, const DeviceParams& dp, int max_N, bool hard, bool soft, bool backward, bool u8,
                               int64_t n_weights, bool again = true);

// Backward of the soft transform through the fast path (every kernel must be a fast-path kernel):
// dW (ragged like the weights, n_weights floats) and db [K] are assigned.
cudaError_t launch_fast_backward(FastState& fs, const DeviceParams& dp, int64_t n_weights, const float* X, int N,
                                 float lambda, float shift, const float* dfeat, const int32_t* argmax, float* dW,
                                 float* db, cudaStream_t stream);

// The launches below return cudaErrorMemoryAllocation, having launched nothing, when there is no room for the copies of one example.
//
// Forward through the fast path: init, pad copy, S kernel, T kernel, finalise.  soft = false:
// PPV + max; soft = true: softPPV + max (+ argmax when argmax != nullptr).
// With X_u8 (raw 8-bit intensities [N][C][L], 4-byte aligned) the samples are normalised per channel
// with *norm while the zero-margined copies are written, and X is not read.  half (hard transform only): samples,
// weights and biases are rounded to binary16 and every multiply-add of the convolution rounds once to binary16.
cudaError_t launch_fast_forward(FastState& fs, const DeviceParams& dp, const float* X, int N, float* feat,
                                cudaStream_t stream, bool soft = false, float lambda = 0.0f, float shift = 0.0f,
                                int32_t* argmax = nullptr, const uint8_t* X_u8 = nullptr, const NormArgs* norm = nullptr,
                                bool half = false);

}  // namespace fast
}  // namespace rocket
