// Host-side launch plan of the fast path: buckets kernels by dilation, lays out band rasters,
// cuts them into tiles and orders the tiles by cost (largest first).
#include <algorithm>
#include <climits>
#include <cmath>
#include <functional>
#include <map>
#include <tuple>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

namespace rocket {
namespace fast {
namespace {

// Clocks of a scheduler: an input row of a tile and channel besides its multiply-adds, a channel, an output row, a tile, a pair, an item;
// clocks of a block: a task.
constexpr double kRRowClocks = 3.0, kRVisitClocks = 30.0, kRPoolClocks = 8.0, kRTileClocks = 120.0, kRPairClocks = 250.0, kRItemClocks = 500.0, kRTaskClocks = 3000.0;

inline int64_t floor_div(int64_t a, int64_t b) { return (a >= 0) ? a / b : -((-a + b - 1) / b); }

// Units of the stream kernel for the kernels whose records start at `first`.  The output rows of a kernel (their count rounded
// up to four) become bands of 16, 12 and 8 rows.  Units of one shape follow one another and within a shape in order of
// dilation, so that the warps running at any one time share an instance of the inner loop and mostly a tensor map.
void build_stream_units(const HostParams& hp, size_t first, int d_max, PlanHost& out) {
    if (first == out.krec.size()) return;
    // Positions a box can reach beyond the samples: three rows before them, seven after (a y step is four rows, of which the
    // last may start three rows further on).  Dilations of random kernels stay below L / 6; handles with larger ones keep the
    // kernel that works on the four copies.
    if (7ll * d_max > 2ll * hp.L + 4096) return;
    out.wfront = (3ll * d_max + 64 + 3) / 4 * 4;
    out.wpitch = (hp.L + std::max<int64_t>(7ll * d_max + 96, out.wfront) + 31) / 32 * 32;
    std::vector<int> order;
    int64_t visits = 0;
    for (size_t f = first; f < out.krec.size(); ++f) {
        const KRec& k = out.krec[f];
        order.push_back((int)f);
        visits += ((int64_t)(k.nout / ((int64_t)16 * k.d)) + 1) * ((k.d + kWarpCols - 1) / kWarpCols) * k.m;
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return out.krec[a].d < out.krec[b].d; });
    // short units where there is little work per warp (148 x 16 of them), so that the warps end together
    const int64_t unit_visits = std::min<int64_t>(kWUnitVisits, std::max<int64_t>(6, visits / (16 * 148 * kWWarps)));
    // Heights for a count of rows (a multiple of four): the fewest rows, where a band costs as much as three rows on top.
    struct Choice { int cost, R; };
    std::vector<Choice> choice(1, {0, 0});
    auto choose = [&](int64_t rows4) {
        while ((int64_t)choice.size() <= rows4) {
            const int t = (int)choice.size();
            Choice best{INT_MAX, 0};
            for (int R : {16, 12, 8}) {
                const int rest = std::max(0, t - R / 4), cost = choice[rest].cost + R + 3;
                if (cost < best.cost) best = {cost, R};
            }
            choice.push_back(best);
        }
        return choice[rows4].R;
    };
    std::map<int, std::vector<WUnit>, std::greater<int>> by_shape;   // longest kernels first, then highest bands
    std::map<std::pair<int, int>, int> map_index;
    for (int fi : order) {
        const KRec& f = out.krec[fi];
        const int64_t tmin = floor_div(f.lo_u, f.d), tmax = floor_div((int64_t)f.hi_u - 1, f.d);
        int64_t rows = (tmax - tmin + 1 + 3) / 4 * 4;
        const int G = w_rows_per_y(f.d), ncol = (f.d + kWarpCols - 1) / kWarpCols;
        for (int64_t t = tmin; rows > 0;) {
            // the bands of the highest kind that pays, all at once
            const int R = choose(std::min<int64_t>(rows, 4096) / 4);
            int64_t n = 1;
            while (rows - n * R > 0 && choose(std::min<int64_t>(rows - n * R, 4096) / 4) == R) ++n;
            out.w_visits += (double)n * ncol * f.m;
            WUnit u{};
            u.krec = fi; u.t0 = (int32_t)t; u.d = f.d; u.m = f.m; u.k = f.k; u.lo_u = f.lo_u; u.hi_u = f.hi_u; u.p = f.p;
            u.tl = f.tl; u.rl = f.rl; u.th = f.th; u.rh = f.rh; u.nout = f.nout; u.woff = f.woff; u.ncol = ncol;
            const int y_rows = (R + f.len - 1 + G - 1) / G;
            const auto found = map_index.emplace(std::make_pair(f.d, y_rows), (int)out.wmaps.size());
            if (found.second) out.wmaps.push_back({f.d, y_rows});
            u.map = found.first->second;
            u.bytes = y_rows * G * kWarpCols * 4;
            u.run = G * f.d;
            u.band_y = R / G;
            u.span = w_span(R, f.d);
            // first row of a y step: the last of its four when they are taken backwards
            const bool backwards = f.d % 4 == 3;
            const int64_t pos = out.wfront + t * f.d + (backwards ? 3ll * f.d : 0);
            u.copy = (int32_t)(pos & 3);
            const int64_t start = pos - u.copy, y = floor_div(start, u.run);
            u.x0 = (int32_t)(start - y * u.run);
            u.y0 = (int32_t)y;
            u.shape = R | f.len << 8 | (backwards ? 3 << 16 : 0);
            for (int q = 0; q < f.m; ++q) u.ch[q] = (uint8_t)f.ch[q];
            std::vector<WUnit>& shape_units = by_shape[(f.len << 8) | R];
            const int64_t tiles = n * ncol, per = std::max<int64_t>(1, unit_visits / f.m), units = (tiles + per - 1) / per;
            for (int64_t i = 0; i < units; ++i) {
                const int64_t beg = tiles * i / units, end = tiles * (i + 1) / units;
                u.tile0 = (int32_t)beg; u.ntiles = (int32_t)(end - beg);
                shape_units.push_back(u);
            }
            rows -= n * R;
            t += n * R;
        }
    }
    size_t total = 0;
    for (auto& kv : by_shape) total += kv.second.size();
    out.wunits.reserve(total);
    for (auto& kv : by_shape) out.wunits.insert(out.wunits.end(), kv.second.begin(), kv.second.end());
}

// The kernels of a handle whose examples fit shared memory.
struct ResidentUnits {
    std::vector<RUnit> units;
    std::vector<double> cost;                          // of a pair, clocks of a scheduler
    double clocks = 0.0, longest = 0.0;
    int tiles = 0;
    int64_t reach = 0;                                 // how far before the first and behind the last sample a tile reads
    double clocks_back[4] = {};                        // the same for each height of the backward
    int64_t reach_back[4] = {};
};

ResidentUnits resident_units(const HostParams& hp, const PlanHost& plan, int kind) {
    const int kHigh = resident_high(kind), kLow = resident_low(kind);
    ResidentUnits out;
    out.units.reserve(plan.krec.size());
    out.cost.reserve(plan.krec.size());
    for (size_t i = 0; i < plan.krec.size(); ++i) {
        const KRec& f = plan.krec[i];
        RUnit u{};
        u.krec = (int32_t)i; u.k = f.k; u.len = f.len; u.d = f.d; u.m = f.m; u.nout = f.nout; u.p = f.p; u.woff = f.woff;
        u.nq = f.nout / f.d; u.nr = f.nout % f.d;
        u.inv_d = 1.0f / (float)f.d;
        const int32_t* S = hp.channel_idx.data() + hp.channel_offset[f.k];
        for (int q = 0; q < f.m; ++q) u.ch[q] = (uint8_t)S[q];
        // bands: all of one height, or as many high ones as fill whole tiles and low ones for the rest, whichever takes least
        const int rows = u.nq + (u.nr > 0 ? 1 : 0);
        auto tiles = [&](int bands) { return ((int64_t)bands * f.d + kWarpCols - 1) / kWarpCols; };
        auto tile_clocks = [&](int R) { return f.m * ((R + f.len - 1) * kRRowClocks + 2.0 * R * f.len + kRVisitClocks) + R * kRPoolClocks + kRTileClocks; };
        const double high = tile_clocks(kHigh), low = tile_clocks(kLow);
        double best = 1e300;
        auto consider = [&](int n) {
            if (n < 0) return;
            const int rest = std::max(0, rows - n * kHigh), n_low = (rest + kLow - 1) / kLow;
            const double c = tiles(n) * high + tiles(n_low) * low;
            if (c < best) { best = c; u.high = n; u.low = n_low; }
        };
        consider((rows + kHigh - 1) / kHigh);
        consider(0);
        for (int64_t t = (int64_t)(rows / kHigh) * f.d / kWarpCols, n = 0; t >= 0 && n < 2; --t, ++n) consider((int)(t * kWarpCols / f.d));
        consider(rows / kHigh);
        const int64_t last_row = (int64_t)u.high * kHigh + u.low * kLow - 1 + f.len - 1;
        out.reach = std::max<int64_t>({out.reach, f.p, last_row * f.d + f.d - f.p - hp.L});
        for (int h = 0; h < 4; ++h) {
            const int R = resident_high(kRBackBands[h]), bands = (rows + R - 1) / R;
            out.clocks_back[h] += tiles(bands) * tile_clocks(R);
            out.reach_back[h] = std::max<int64_t>({out.reach_back[h], f.p, (int64_t)(bands * R + f.len - 2) * f.d + f.d - f.p - hp.L});
        }
        out.tiles = (int)std::max<int64_t>(out.tiles, tiles(u.high) + tiles(u.low));
        best += kRPairClocks;
        out.clocks += best / 4.0;
        out.longest = std::max(out.longest, best);
        out.units.push_back(u);
        out.cost.push_back(best);
    }
    return out;
}

void build_resident_units(const HostParams& hp, PlanHost& out) {
    const int64_t row = (hp.L + 3ll) / 4 * 4;
    if (hp.C * row > kRMostFloats || hp.L > kRMostSteps) return;
    const int64_t room = (kRMostFloats - hp.C * row) / (hp.C + 1) / 4 * 4;   // for zeros around the rows
    int32_t most_padding = 0;
    for (const KRec& f : out.krec) {
        if (f.nout > kRMostOutputs || f.d > kRMostOutputs) return;
        most_padding = std::max(most_padding, f.p);
    }
    if (hp.L > kRMostStepsTested && room < most_padding) return;
    ResidentUnits r = resident_units(hp, out, 0);
    if (hp.L <= kRTallSteps) {
        const int other = hp.L < kRSmallSteps ? 1 : 2;
        ResidentUnits s = resident_units(hp, out, other);
        if (s.clocks < r.clocks) {
            out.r_bands = other;
            r = std::move(s);
        }
    }
    out.r_clocks = r.clocks;
    out.r_longest = r.longest;
    out.r_tiles = r.tiles;
    const int64_t most_zeros = std::min(room, 2 * row);
    int h = 0;
    for (int other = 1; other < 4; ++other)
        if (r.reach_back[h] > most_zeros || (r.reach_back[other] <= most_zeros && r.clocks_back[other] < r.clocks_back[h])) h = other;
    const bool back = r.reach_back[h] <= most_zeros;
    // Zeros around the rows make all reads alike; where they would not fit, or take more than twice the samples, some tiles test theirs.
    const int zeros = (int)std::min((std::max(r.reach, back ? r.reach_back[h] : 0) + 3) / 4 * 4, most_zeros);
    out.r_front = zeros;
    out.r_pitch = (int)row + zeros;
    out.r_zeros = zeros >= r.reach;
    out.resident = !r.units.empty() && hp.L <= (out.r_zeros ? kRMostSteps : kRMostStepsTested);
    if (!out.resident) return;
    out.r_back = back ? kRBackBands[h] : 0;
    const bool far = hp.L > kRTilesFarSteps;
    if (hp.L >= kRTilesSteps && hp.C >= (far ? 2 : hp.L <= kRTilesMidSteps ? 3 : 6) && hp.C <= kSMaxPlanes && (int)out.krec.size() >= kRTilesKernels)
        out.r_tiles_from = (int)std::ceil((far ? kRTilesFarPairs : kRTilesPairs) / (double)out.krec.size());
    for (RUnit& u : r.units) {
        const int before = std::max(0, u.p - zeros), end = hp.L + u.p + zeros;
        u.pq = before / u.d; u.pr = before % u.d;
        u.lq = end / u.d; u.lr = end % u.d;
    }
    // Kernels of a length follow one another, so that the warps of a block share inner loops; the longest pairs of a length first.  The
    // instruction caches decide here: the longest pairs first throughout take 548 us where this order takes 222 (24 x 32 x 1,751, 2,000 kernels).
    std::vector<int> order(r.units.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return r.units[a].len != r.units[b].len ? r.units[a].len > r.units[b].len : r.cost[a] > r.cost[b];
    });
    out.runits.reserve(order.size());
    for (int i : order) out.runits.push_back(r.units[i]);
}

}  // namespace

// Blocks take tasks of a few examples and a part of the kernels: as few copies of an example as leave every SM its share.
ResidentSplit resident_split(const PlanHost& plan, int N, int C, int sms, int mode) {
    const double work = plan.r_clocks * (mode == 1 ? 1.4 : mode == 2 ? 2.6 : 1.0);
    const int64_t n_units = (int64_t)plan.runits.size();
    const int warps = resident_warps(mode, mode == 2 ? plan.r_back : plan.r_bands);
    // eight items per warp and task, if that many there are
    auto run_of = [&](int64_t kernels, int64_t e) { return std::max<int64_t>(1, std::min<int64_t>(e, kernels * e / (8 * warps))); };
    ResidentSplit best{1, N, 1, 1, 1, 1u};
    double least = 1e300;
    for (int64_t e = 1; e <= N && resident_floats(plan, e, C) <= kRMostFloats; e *= 2) {
        const int64_t groups = (N + e - 1) / e;
        int64_t last = 0;
        for (int64_t rounds = 1; rounds <= 64; ++rounds) {
            const int64_t parts = std::min(n_units, rounds * sms / groups);
            if (parts < 1 || parts == last) continue;
            last = parts;
            const int64_t kernels = (n_units + parts - 1) / parts, run = run_of(kernels, e);
            for (int split = 1; split <= 4 && (split == 1 || (run == 1 && split < 2 * plan.r_tiles)); split *= 2) {
                if (resident_floats(plan, e, C) + resident_merge_floats(plan, e, (int)parts, split, mode) > kRMostFloats) continue;
                const double items = (double)kernels * (double)((e + run - 1) / run) * split;
                // a warp's last item runs beside those of the four to six other warps of its scheduler
                const double task = kRTaskClocks + 4.0 * e * C * plan.r_pitch / 30.0 + e * work / parts + items * kRItemClocks / 4.0 +
                                    2.0 * plan.r_longest * (double)run / std::min(split, plan.r_tiles);
                const double t = (double)((groups * parts + sms - 1) / sms) * task;
                if (t < least) { least = t; best = {(int)e, (int)groups, (int)parts, (int)run, split, 1u}; }
            }
        }
    }
    best.grid = (unsigned)std::min<int64_t>((int64_t)best.groups * best.parts, sms);
    return best;
}

// One example where a bucket has many kernels, up to 4 and up to 16 where it has some or few (64 to 256 pairs per tile for its 16
// warps), as far as the planes hold them and the launch keeps two tiles per SM.
SGroups s_groups(const PlanHost& plan, int N, int sms) {
    const int fit = (plan.s_wide ? kSWidePlanes : kSMaxPlanes) / std::max(1, plan.s_max_nch);
    SGroups a{};
    unsigned long long tiles = 0;
    for (int shift = 0; shift < 5; ++shift) {
        tiles = 0;
        for (int cls = 0; cls < 3; ++cls) {
            const int most = cls == 0 ? 1 : cls == 1 ? 4 : 16;
            a.end[cls] = plan.s_class_end[cls];
            a.examples[cls] = std::max(1, std::min({fit, most, N}) >> shift);
            a.groups[cls] = (N + a.examples[cls] - 1) / a.examples[cls];
            tiles += (unsigned long long)(a.end[cls] - (cls ? a.end[cls - 1] : 0)) * a.groups[cls] * (plan.s_wide ? 2 : 1);
        }
        if (tiles >= 2ull * sms || a.examples[2] == 1) break;
    }
    a.grid = (unsigned)std::min<unsigned long long>(tiles, (unsigned long long)sms);
    return a;
}

int stream_chunk(int C, int64_t pitch) {
    const int64_t example = 4 * kWCopies * (int64_t)C * pitch;
    const int64_t few = std::max<int64_t>(1, std::min<int64_t>(kWFewExamples, kWMostCopyBytes / example));
    return (int)std::min<int64_t>(1 << 16, std::max<int64_t>(few, kWCopyBytes / example));
}

// Examples of an item: as many as give it kWItemVisits visits on average, while every warp of the chip still gets a dozen items and
// their copies take no more than half of the L2: two examples of 20 x 200,000 do not, and 60 of them took 245 ms two at a time, 218
// one at a time (10,000 kernels; 20 x 100,000: 106 and 103 ms; 20 x 50,000, where two fit: 50.7 and 51.6).
// Groups of a set: as many as keep their copies in a third of the L2.  The soft transform and the backward take more of them where a
// handle has few units: in the course of a set the warps pass through all nine shapes of the inner loop, and with fewer than
// kWSoftSetItems items per warp they wait for instructions (24 x 12 x 50,000, 340 kernels, both passes: 8.68 ms by bytes alone,
// 7.44, 6.46, 6.40 and 6.40 with 4, 8, 16 and 24 items; 24 x 20 x 14,002, 1,200 kernels: 6.32 and 4.56).  The hard modes, whose code
// is smaller, lose by it (24 x 12 x 50,000, 340 kernels: 1.91 and 2.06).
StreamItems stream_items(int N, int C, int L, int n_units, double visits, int mode, int sms, int64_t l2_bytes) {
    StreamItems s;
    const int64_t warps = (int64_t)sms * kWWarps, example_bytes = (int64_t)C * kWCopies * L * 4;
    const double per_unit = std::max(1.0, visits * (mode == 2 ? 2.0 : 1.0) / std::max(1, n_units));
    s.examples = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)(kWItemVisits / per_unit), (int64_t)N * n_units / (warps * 12), (int64_t)N,
                                                              l2_bytes / 2 / example_bytes}));
    s.groups = (N + s.examples - 1) / s.examples;
    int64_t per_set = l2_bytes / 3 / (example_bytes * s.examples);
    if (mode == 1 || mode == 2) per_set = std::max(per_set, (kWSoftSetItems * warps + n_units - 1) / std::max(1, n_units));
    s.groups_per_set = (int)std::max<int64_t>(1, std::min<int64_t>(s.groups, per_set));
    return s;
}

namespace {

// Costs for generic_pays, fitted to the device times of 570 calls of 21 to 255 channels, 24 to 20,000 steps, 30 to 5,000 kernels and
// 1 to 128 examples (9 % rms on either side).  The costs are the hard transform's; training takes 3.1 times as long through the fused
// kernels and 3.4 times through the generic ones.
constexpr double kUsFused = 6.2, kUsStream = 6.0, kUsTile = 3.25, kUsPlane = 0.159, kUsTap = 0.0112, kUsVisit = 5.9e-4, kUsCopiedByte = 1.28e-7;
constexpr double kUsGeneric = 1.9, kUsPair = 2.2e-3, kUsWarpTap = 8.35e-6, kUsBlockTap = 8.2e-5, kUsTapLatency = 0.0696;
constexpr double kSoftGeneric = 3.4 / 3.1, kNearTie = 1.03;    // within the error of the estimates the fused kernels have it

void estimate_costs(const HostParams& hp, PlanHost& p) {
    const double halves = p.s_wide ? 2.0 : 1.0, plane = kUsPlane * (p.s_wide ? 23.0 / 34.0 : 1.0);
    std::vector<double> taps(p.sb.size(), 0.0);
    for (size_t b = 0; b < p.sb.size(); ++b)
        for (int f = p.sb[b].kbeg; f < p.sb[b].kend; ++f) taps[b] += (double)p.krec[f].m * p.krec[f].len;
    double most = -1.0;
    for (const SItem& it : p.sitems) {
        const double tile = kUsTile + p.sb[it.bucket].nch * plane, work = taps[it.bucket] * kUsTap;
        p.us_s += halves * tile + work;
        if (work > most) {                                     // the longest tile, not the widest
            most = work;
            p.us_s_tile = tile + work / halves;
        }
    }
    double visits = p.w_visits;
    int64_t row_bytes = p.wunits.empty() ? 0 : 4 * kWCopies * p.wpitch;
    for (const TItem& it : p.titems) visits += (double)it.m * kTConsumerWarps;
    if (p.wunits.empty() && !p.titems.empty()) row_bytes = 4 * 4 * p.pad_pitch;
    p.us_t = visits * kUsVisit + (double)hp.C * row_bytes * kUsCopiedByte;
    for (int k = 0; k < hp.K; ++k) {
        const int64_t nout = (int64_t)hp.L + 2 * (int64_t)hp.padding[k] - (int64_t)(hp.length[k] - 1) * hp.dilation[k];
        const double t = (double)hp.length[k] * hp.num_channels[k], rounds = t * (double)((nout + 255) / 256);
        p.us_g += kUsPair + kUsWarpTap * t * (double)((nout + 31) / 32) + kUsBlockTap * rounds;
        p.us_g_kernel = std::max(p.us_g_kernel, kUsTapLatency * rounds);
    }
}

// Rows of the S bands: the height that takes the fewest clocks over all tiles.  A tile costs 3,000 clocks and its copies (24 B/clk) besides the
// work of its kernels; a low band reads more rows per row of outputs, a high one may leave a dilation's last tile half empty (20 x 5,000: 81 % of the
// positions of tiles of 24 rows are outputs, 89 % of 21).  Measured (us, 24 rows and the chosen height): 64 x 20 x 5,000 and 10,000 kernels 6,173
// and 5,923, 1 x 20 x 5,000 322 and 289, backward of 24 x 20 x 5,000 and 3,000 kernels 2,087 and 1,948.
int s_band_rows(const HostParams& hp, const std::vector<std::pair<int, std::vector<int>>>& groups) {
    struct Sums { int64_t d, tmin, tmax; double taps, visits, kernels; int nch; };   // taps: products per output; visits: (kernel, channel) pairs
    std::vector<Sums> sums;
    for (const auto& kv : groups) {
        Sums g{kv.first, INT64_MAX, INT64_MIN, 0.0, 0.0, (double)kv.second.size(), 0};
        std::vector<char> used(hp.C, 0);
        int64_t lo = INT64_MAX, hi = INT64_MIN;
        for (int k : kv.second) {
            const int len = hp.length[k], m = hp.num_channels[k];
            lo = std::min<int64_t>(lo, -(int64_t)hp.padding[k]);
            hi = std::max<int64_t>(hi, (int64_t)hp.L + hp.padding[k] - (len - 1) * g.d);
            g.taps += (double)m * len;
            g.visits += m;
            for (int q = hp.channel_offset[k]; q < hp.channel_offset[k] + m; ++q)
                if (!used[hp.channel_idx[q]]) { used[hp.channel_idx[q]] = 1; ++g.nch; }
        }
        g.tmin = floor_div(lo, g.d);
        g.tmax = floor_div(hi - 1, g.d);
        sums.push_back(g);
    }
    int best_rows = kRS;
    double best = 1e300;
    for (int R : {kRS, kSLowRows[0], kSLowRows[1]}) {
        double clocks = 0.0;
        for (const Sums& g : sums) {
            const double work = (2.0 * R + 1.5) * g.taps + (1.5 * R + 40.0) * g.visits + (8.0 * R + 120.0) * g.kernels;
            const int64_t bands = (g.tmax - g.tmin + R) / R, tiles = (bands * g.d + kWarpCols - 1) / kWarpCols;
            clocks += (double)tiles * (work / 4.0 + 3000.0 + g.nch * (R + 10) * kWarpCols * 4 / 24.0);
        }
        if (clocks < 0.99 * best) { best = clocks; best_rows = R; }
    }
    return best_rows;
}

}  // namespace

// A series of more channels than a tile has planes for needs buckets and copies that few or short kernels do not pay for: the generic
// kernels, which read what a kernel uses and no more, take 14 us for 1 x 32 x 32 and 1,500 kernels where the fused ones take 140,
// 71 us for 32 x 255 x 1,002 and 60 kernels against 113; from some 500 steps on the fused ones are ahead (24 x 32 x 1,751, 2,000
// kernels: 1,445 us against 477).
bool generic_pays(const PlanHost& plan, int N, int sms, bool soft) {
    // a launch lasts as long as its work for the SMs or its longest block, whichever is more, and near a tie somewhat longer than both;
    // the generic kernels' blocks, as long as their kernels' outputs, pack worse
    auto both = [](double work, double longest, double q) { return std::pow(std::pow(work, q) + std::pow(longest, q), 1.0 / q); };
    const double fused = kUsFused + both(N * plan.us_s / sms, plan.us_s_tile, 4.0) + (plan.us_t > 0.0 ? kUsStream : 0.0) + N * plan.us_t;
    const double generic = kUsGeneric + both(N * plan.us_g, plan.us_g_kernel, 1.5);
    return kNearTie * (soft ? kSoftGeneric : 1.0) * generic < fused;
}

int pays_up_to(const PlanHost& plan, int max_N, int sms, bool soft, bool generic) {
    if (generic_pays(plan, max_N, sms, soft) == generic) return max_N;
    for (int n = 1 << 16; n >= 1; n /= 2)
        if (n < max_N && generic_pays(plan, n, sms, soft) == generic) return std::min(max_N, 2 * n - 1);
    return 0;
}

void fill_record_weights(const HostParams& hp, KRec& f) {
    const float* W = hp.weights.data() + hp.weight_offset[f.k];
    f.negb = 0.0f - hp.bias[f.k];
    for (int q = 0; q < f.m; ++q)
        for (int j = 0; j < f.len; ++j) f.w2[q][2 * j] = f.w2[q][2 * j + 1] = 0.0f - W[q * f.len + j];
}

void build_plan(const HostParams& hp, int split, PlanHost& out, bool all_tiles, bool only_used) {
    out = PlanHost();
    out.flops_s = out.flops_t = 0.0;
    if (split < kTMinDilation) split = kTMinDilation;
    const int K = hp.K;
    // Short series: where every dilation is below 128 the S kernel takes them all, which saves the staging copy and a
    // launch for a handful of kernels (16 x 1 x 512, 1,000 kernels: 124 -> 90 us).
    {
        int d_top = 0;
        for (int k = 0; k < K; ++k) d_top = std::max(d_top, hp.dilation[k]);
        if (d_top < 2 * kTMinDilation) split = std::max(split, 2 * kTMinDilation);
    }
    out.split = split;
    // Any series length will do: the small-dilation kernel copies single floats and the large-dilation kernel reads the
    // zero-margined copies, whose pitch does not depend on L.
    const bool shape_ok = hp.C <= kMaxChannels && hp.L >= 16;
    std::vector<int> s_kernels, t_kernels;
    for (int k = 0; k < K; ++k) {
        const int len = hp.length[k], d = hp.dilation[k];
        const bool fast_len = (len == 7 || len == 9 || len == 11);
        if (!shape_ok || !fast_len) out.generic_list.push_back(k);
        else if (d < split) s_kernels.push_back(k);
        else t_kernels.push_back(k);
    }
    out.enabled = !(s_kernels.empty() && t_kernels.empty());
    if (!out.enabled) return;

    out.krec.reserve(s_kernels.size() + t_kernels.size());
    auto add_kernel = [&](int k) {
        out.krec.emplace_back();
        KRec& f = out.krec.back();
        f.len = hp.length[k]; f.d = hp.dilation[k]; f.p = hp.padding[k]; f.m = hp.num_channels[k];
        f.nout = (int32_t)((int64_t)hp.L + 2 * (int64_t)f.p - (int64_t)(f.len - 1) * f.d);
        f.k = k; f.lo_u = -f.p; f.hi_u = f.nout - f.p;
        f.woff = hp.weight_offset[k];
        f.tl = (int32_t)floor_div(f.lo_u, f.d); f.rl = f.lo_u - f.tl * f.d;
        f.th = (int32_t)floor_div(f.hi_u, f.d); f.rh = f.hi_u - f.th * f.d;
        const int32_t* S = hp.channel_idx.data() + hp.channel_offset[k];
        for (int q = 0; q < f.m; ++q) f.ch[q] = S[q];
        fill_record_weights(hp, f);
    };

    if (only_used && (int64_t)hp.C * hp.L <= kRMostFloats && hp.L <= kRMostSteps) {
        // series for which the resident kernel most likely serves every pass: then nothing else is needed
        for (const auto* list : {&s_kernels, &t_kernels})
            for (int k : *list) {
                add_kernel(k);
                const KRec& f = out.krec.back();
                (list == &s_kernels ? out.flops_s : out.flops_t) += 2.0 * f.len * f.m * (double)f.nout;
            }
        build_resident_units(hp, out);
        if (resident_backward(out) && out.r_tiles_from == 0) return;
        out.krec.clear();
        out.runits.clear();
        out.resident = false;
        out.r_back = out.r_tiles_from = 0;
        out.flops_s = out.flops_t = 0.0;
    }

    // ---- S regime: one bucket per dilation, kernels inside ordered by cost (largest first: the warps of a
    // block pull them one by one, so the cheap ones fill the end of a tile evenly).  Buckets with many
    // kernels per warp are ordered by length first: warps that run side by side then share one instance of
    // the inner loops, which the instruction caches reward (backward 5 % faster, hard transform unchanged;
    // for the small buckets the balance at the end of a tile is worth more).
    std::map<int, std::vector<int>> by_d;
    for (int k : s_kernels) by_d[hp.dilation[k]].push_back(k);
    struct Cost { double c; int idx; };
    std::vector<Cost> s_cost;
    // Kernels of one dilation that use more channels than a tile has planes are split: a kernel (most channels
    // first) joins the group whose channel set grows least, or opens a new one.
    std::vector<std::pair<int, std::vector<int>>> groups;
    std::map<int, int> channels_of;
    for (const auto& kv : by_d) {
        std::vector<char> used(hp.C, 0);
        int& n_used = channels_of[kv.first];
        for (int k : kv.second)
            for (int q = hp.channel_offset[k]; q < hp.channel_offset[k] + hp.num_channels[k]; ++q)
                if (!used[hp.channel_idx[q]]) { used[hp.channel_idx[q]] = 1; ++n_used; }
    }
    {   // halves where that lets every dilation be one bucket; two of 34 channels are no better than several of 20 (64 channels)
        int most = 0;
        for (const auto& c : channels_of) most = std::max(most, c.second);
        out.s_wide = most > kSMaxPlanes && most <= kSWidePlanes;
    }
    const int max_planes = out.s_wide ? kSWidePlanes : kSMaxPlanes;
    for (auto& kv : by_d) {
        if (channels_of[kv.first] <= max_planes) {
            groups.emplace_back(kv.first, std::move(kv.second));
            continue;
        }
        std::stable_sort(kv.second.begin(), kv.second.end(), [&](int a, int b) { return hp.num_channels[a] > hp.num_channels[b]; });
        struct Group { std::vector<char> has; int n; std::vector<int> ks; };
        std::vector<Group> gs;
        for (int k : kv.second) {
            const int32_t* S = hp.channel_idx.data() + hp.channel_offset[k];
            int best = -1, best_new = INT_MAX;
            for (size_t g = 0; g < gs.size(); ++g) {
                int fresh = 0;
                for (int q = 0; q < hp.num_channels[k]; ++q) fresh += !gs[g].has[S[q]];
                if (gs[g].n + fresh <= max_planes && fresh < best_new) { best = (int)g; best_new = fresh; }
            }
            if (best < 0) { best = (int)gs.size(); gs.push_back({std::vector<char>(hp.C, 0), 0, {}}); }
            Group& g = gs[best];
            for (int q = 0; q < hp.num_channels[k]; ++q)
                if (!g.has[S[q]]) { g.has[S[q]] = 1; ++g.n; }
            g.ks.push_back(k);
        }
        for (Group& g : gs) groups.emplace_back(kv.first, std::move(g.ks));
    }
    if (!all_tiles && hp.C <= kSMaxPlanes) out.s_rows = s_band_rows(hp, groups);
    const int band_rows = out.s_rows;
    for (auto& kv : groups) {
        const int d = kv.first;
        auto& ks = kv.second;
        std::stable_sort(ks.begin(), ks.end(), [&](int a, int b) {
            if ((int)ks.size() >= kSLengthOrderMin && hp.length[a] != hp.length[b]) return hp.length[a] > hp.length[b];
            return hp.length[a] * hp.num_channels[a] > hp.length[b] * hp.num_channels[b];
        });
        SBucket b{};
        b.d = d; b.kbeg = (int32_t)out.krec.size();
        int64_t tmin = INT64_MAX, tmax = INT64_MIN;
        int maxlen = 0;
        double work = 0.0;
        for (int k : ks) {
            add_kernel(k);
            const KRec& f = out.krec.back();
            out.flops_s += 2.0 * f.len * f.m * (double)f.nout;
            tmin = std::min(tmin, floor_div(f.lo_u, d));
            tmax = std::max(tmax, floor_div((int64_t)f.hi_u - 1, d));
            maxlen = std::max(maxlen, f.len);
            work += (double)f.m * (f.len + 2) + 6.0;
        }
        b.kend = (int32_t)out.krec.size();
        {   // the bucket's channel list; the records get positions in it
            std::vector<int> at(hp.C, -1);
            for (int f = b.kbeg; f < b.kend; ++f)
                for (int q = 0; q < out.krec[f].m; ++q) at[out.krec[f].ch[q]] = 0;
            for (int c = 0; c < hp.C; ++c)
                if (at[c] == 0) { b.ch[b.nch] = (uint8_t)c; at[c] = b.nch++; }
            for (int f = b.kbeg; f < b.kend; ++f)
                for (int q = 0; q < out.krec[f].m; ++q) out.krec[f].ch[q] = at[out.krec[f].ch[q]];
            out.s_max_nch = std::max(out.s_max_nch, b.nch);
        }
        b.tmin = (int32_t)tmin;
        b.nbands = (int32_t)((tmax - tmin + 1 + band_rows - 1) / band_rows);
        b.raster_len = b.nbands * d;
        b.rows = band_rows + maxlen - 1;
        const int bi = (int)out.sb.size();
        out.sb.push_back(b);
        // a tile is interior when its 64 raster positions exist and the u of every (row, column) lies inside
        // the output range of every kernel of the bucket
        int64_t lo_max = INT64_MIN, hi_min = INT64_MAX;
        for (int f = b.kbeg; f < b.kend; ++f) {
            lo_max = std::max<int64_t>(lo_max, out.krec[f].lo_u);
            hi_min = std::min<int64_t>(hi_min, out.krec[f].hi_u);
        }
        for (int c0 = 0; c0 < b.raster_len; c0 += kWarpCols) {
            bool interior = c0 + kWarpCols <= b.raster_len;
            for (int c = c0; interior && c < c0 + kWarpCols; ++c) {
                const int64_t u0 = s_column_u0(b, c, band_rows);
                interior = u0 >= lo_max && u0 + (int64_t)(band_rows - 1) * d < hi_min;
            }
            s_cost.push_back({work + 0.3 * b.nch * b.rows, (int)out.sitems.size()});
            out.sitems.push_back({bi, c0, interior ? 1 : 0, 0});
        }
    }
    {
        std::stable_sort(s_cost.begin(), s_cost.end(), [](const Cost& a, const Cost& b) { return a.c > b.c; });
        std::vector<SItem> sorted;
        sorted.reserve(out.sitems.size());
        for (int cls = 0; cls < 3; ++cls) {
            for (auto& c : s_cost) {
                const SBucket& b = out.sb[out.sitems[c.idx].bucket];
                const int n = b.kend - b.kbeg;
                if ((n >= kSManyKernels ? 0 : n >= kSSomeKernels ? 1 : 2) == cls) sorted.push_back(out.sitems[c.idx]);
            }
            out.s_class_end[cls] = (int)sorted.size();
        }
        out.sitems.swap(sorted);
    }

    // ---- T regime: per kernel, the grid of 16-row x 64-column warp tiles is cut into block tiles of
    // rg x cg warp tiles (rg * cg <= the consumer warps of a block); the column-group width that needs the
    // fewest block tiles wins
    int d_max = 0;
    std::map<std::tuple<int, int, int>, int> map_index;
    // kernels of one length follow one another, so that the blocks running at any one time execute the same
    // instance of the inner loops (instruction caches: backward 3.5 % faster, forward 0.1-1 %); within a length by
    // dilation, whose tile shapes decide which instance it is (backward another 2 %: 74.0 -> 72.5 ms at 32 x 20 x 50,000)
    std::stable_sort(t_kernels.begin(), t_kernels.end(), [&](int a, int b) {
        return hp.length[a] != hp.length[b] ? hp.length[a] > hp.length[b] : hp.dilation[a] < hp.dilation[b];
    });
    const size_t first_t = out.krec.size();
    for (int k : t_kernels) {
        add_kernel(k);
        const KRec& f = out.krec.back();
        out.flops_t += 2.0 * f.len * f.m * (double)f.nout;
        d_max = std::max(d_max, f.d);
    }
    build_stream_units(hp, first_t, d_max, out);
    // the tiles are for handles without stream units (a third of the time to make a handle of 10,000 kernels)
    const size_t end_t = all_tiles || out.wunits.empty() ? out.krec.size() : first_t;
    for (size_t ki = first_t; ki < end_t; ++ki) {
        const KRec& f = out.krec[ki];
        const int64_t tmin = floor_div(f.lo_u, f.d);
        const int64_t tmax = floor_div((int64_t)f.hi_u - 1, f.d);
        const int R16 = (int)((tmax - tmin + 1 + kR - 1) / kR), C64 = (f.d + kWarpCols - 1) / kWarpCols;
        // column chunks for a main width cg: C64 / cg chunks of cg, the rest in chunks of 2 and 1
        auto chunks_of = [&](int cg, std::vector<int>& widths) {
            widths.assign(C64 / cg, cg);
            int rest = C64 % cg;
            if (rest >= 2) { widths.push_back(2); rest -= 2; }
            if (rest >= 1) widths.push_back(1);
        };
        constexpr int W = kTConsumerWarps;
        // A single row group under tiles narrower than the block has warps would leave warps idle: it can be cut
        // into wide tiles instead (all consumer warps side by side, only the rows that hold samples), as long
        // as the halves fit a stage.
        auto wide_fits = [&](int r16) {
            const TWindow win = t_window((int)(tmin + (int64_t)kR * r16), kR + f.len - 1, f.d, hp.L);
            return C64 > W / 2 && kTWideHalves * t_wide_half_floats(win.g_hi - win.g_lo) <= kTStageFloats;
        };
        // widths of the tiles of a wide band: W column groups each, the rest in ordinary tiles of one row group
        std::vector<int> wide_widths(C64 / W, W);
        {
            int rest = C64 % W;
            if (rest > W / 2) { wide_widths.push_back(W); rest = 0; }
            if (W > 4 && rest >= 3) { wide_widths.push_back(4); rest = 0; }
            if (rest >= 2) { wide_widths.push_back(2); rest -= 2; }
            if (rest >= 1) wide_widths.push_back(1);
        }
        // candidates: main width 2, 4 or 1 over all row groups, or the widest main width over all row groups
        // but the last and wide tiles over that one; the fewest block tiles win
        int best_cg = 2;
        bool last_wide = false;
        int64_t best_tiles = INT64_MAX;
        for (int cg : {2, 4, 1}) {
            if (cg > kTMaxCg) continue;
            std::vector<int> widths;
            chunks_of(cg, widths);
            int64_t tiles = 0;
            for (int w : widths) tiles += (R16 + W / w - 1) / (W / w);
            if (tiles < best_tiles) { best_tiles = tiles; best_cg = cg; }
        }
        if (R16 % 2 == 1 && wide_fits(R16 - 1)) {
            std::vector<int> widths;
            chunks_of(kTMaxCg, widths);
            int64_t tiles = (int64_t)wide_widths.size();
            for (int w : widths) tiles += (R16 - 1 + W / w - 1) / (W / w);
            if (tiles < best_tiles) { best_tiles = tiles; best_cg = kTMaxCg; last_wide = true; }
        }
        struct Band { int r16, nrg; std::vector<int> widths; bool wide_band; };
        std::vector<Band> bands;
        std::vector<int> main_widths;
        chunks_of(best_cg, main_widths);
        const int main_rows = last_wide ? R16 - 1 : R16;
        if (main_rows > 0) bands.push_back({0, main_rows, main_widths, false});
        if (last_wide) bands.push_back({R16 - 1, 1, wide_widths, true});
        for (const Band& band : bands) {
            int c64 = 0;
            for (int w : band.widths) {
                const bool wide_tile = band.wide_band && w == W;
                const int rg_full = wide_tile ? 1 : W / w;
                for (int r16 = band.r16; r16 < band.r16 + band.nrg; r16 += rg_full) {
                    TItem it{};
                    it.rg = std::min(rg_full, band.r16 + band.nrg - r16);
                    it.wide = wide_tile ? 1 : 0;
                    it.cg = it.wide ? 4 : w;
                    it.t0 = (int32_t)(tmin + (int64_t)kR * r16); it.r0 = c64 * kWarpCols;
                    // a tile none of whose (row, column) pairs is an output of the kernel is left out
                    bool any_output = false;
                    for (int t = it.t0; t < it.t0 + kR * it.rg && !any_output; ++t) {
                        const int64_t c_lo = std::max<int64_t>(it.r0, (int64_t)f.lo_u - (int64_t)t * f.d);
                        const int64_t c_hi = std::min<int64_t>(std::min(it.r0 + kWarpCols * w, f.d), (int64_t)f.hi_u - (int64_t)t * f.d);
                        any_output = c_lo < c_hi;
                    }
                    if (!any_output) continue;
                    it.d = f.d; it.len = f.len; it.m = f.m;
                    const TWindow win = t_window(it.t0, kR + f.len - 1, f.d, hp.L);
                    it.g_lo = it.wide ? win.g_lo : 0;
                    it.g_hi = it.wide ? win.g_hi : t_box_rows(it.rg, f.len);
                    it.box_rows = it.g_hi - it.g_lo;
                    for (int q = 0; q < f.m; ++q) it.ch[q] = (uint8_t)f.ch[q];
                    it.krec = (int)ki;
                    const auto key = std::make_tuple(f.d, t_box_cols(it.cg), it.box_rows);
                    auto found = map_index.find(key);
                    if (found == map_index.end()) {
                        found = map_index.emplace(key, (int)out.tmaps.size()).first;
                        out.tmaps.push_back({f.d, t_box_cols(it.cg), it.box_rows});
                    }
                    it.map = found->second;
                    // per consumer warp: does every / any (row, column) of its warp tile hold an output?
                    for (int w8 = 0; w8 < kTConsumerWarps; ++w8) {
                        const int wr = it.wide ? 0 : w8 / it.cg, wc = it.wide ? w8 : w8 % it.cg;
                        if (wr >= it.rg) continue;
                        const int64_t ta = (int64_t)it.t0 + kR * wr, ca = (int64_t)it.r0 + kWarpCols * wc;
                        const int64_t cb = std::min<int64_t>(ca + kWarpCols, f.d);
                        if (cb <= ca) continue;
                        bool any = false;
                        for (int64_t t = ta; t < ta + kR && !any; ++t)
                            any = std::max<int64_t>(t * f.d + ca, f.lo_u) < std::min<int64_t>(t * f.d + cb, f.hi_u);
                        if (any) it.warp_active |= 1 << w8;
                        if (cb == ca + kWarpCols && ta * f.d + ca >= f.lo_u && (ta + kR - 1) * f.d + cb - 1 < f.hi_u)
                            it.warp_interior |= 1 << w8;
                    }
                    for (int ph = 0; ph < 4; ++ph) {
                        const TPhase tp = t_phase(it.t0, it.r0, it.d, ph);
                        it.x[ph] = tp.x; it.y[ph] = tp.y + it.g_lo; it.j[ph] = tp.j;
                    }
                    out.titems.push_back(it);
                }
                c64 += w;
            }
        }
    }
    // every channel row of the zero-margined copy: front zeros, L samples, zeros for the run a box may
    // read past the last sample; rounded to 128 bytes
    const int64_t pitch = (int64_t)kTPadFront + hp.L + 4ll * d_max + kTXExtra + t_box_cols(4);
    out.pad_pitch = (pitch + 31) / 32 * 32;
    if (hp.C > kSMaxPlanes) estimate_costs(hp, out);
    build_resident_units(hp, out);
}

}  // namespace fast
}  // namespace rocket
