// Host-side check of the resident kernel's plan (no GPU needed): replays, with the kernel's own column arithmetic, which outputs the
// lanes of every tile own and which samples (or zeros around them) they read, and how calls are dealt to blocks.  Every output of every kernel is owned once,
// every input row counted as a sample lies in the series (and no other one does), every example and kernel is dealt once.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

using namespace rocket;
using namespace rocket::fast;

namespace rocket { std::atomic<int64_t> g_launch_count{0}; }

#define REQUIRE(cond, ...)                                        \
    do {                                                          \
        if (!(cond)) {                                            \
            std::fprintf(stderr, "FAIL %s:%d: ", __FILE__, __LINE__); \
            std::fprintf(stderr, __VA_ARGS__);                    \
            std::fprintf(stderr, "\n");                           \
            std::exit(1);                                         \
        }                                                         \
    } while (0)

// backward: in the bands of its own, all of whose reads are samples or zeros
static void check_units(const PlanHost& plan, int L, bool backward) {
    const int bands = backward ? plan.r_back : plan.r_bands;
    const bool one_height = resident_high(bands) == resident_low(bands);
    for (const RUnit& u : plan.runits) {
        std::vector<int> owned(u.nout, 0);
        for (int half = 0; half < 2; ++half) {
            const int high = resident_high(bands), R = half ? resident_low(bands) : high;
            const int high_bands = one_height ? (u.nq + (u.nr > 0) + high - 1) / high : u.high, low_bands = one_height ? 0 : u.low;
            const int ncols = (half ? low_bands : high_bands) * u.d, base = half ? high * high_bands : 0;
            for (int c0 = 0; c0 < ncols; c0 += kWarpCols)
                for (int l = 0; l < kWarpCols; ++l) {
                    const int c = std::min(c0 + l, ncols - 1);
                    const ResidentColumn at = resident_column(u, c, base, R);
                    REQUIRE(at.band == c / u.d, "band of column %d at dilation %d", c, u.d);
                    const int rows = R + u.len - 1, out = c0 + l < ncols ? at.out : 0;
                    for (int o = 0; o < out; ++o) {
                        const int64_t i = at.i0 + (int64_t)o * u.d;
                        REQUIRE(i >= 0 && i < u.nout, "output %lld of %d", (long long)i, u.nout);
                        ++owned[i];
                    }
                    if (out < R && c0 + l < ncols) REQUIRE(at.i0 + (int64_t)out * u.d >= u.nout, "an output is left out");
                    for (int s = 0; s < rows; ++s) {
                        const int64_t x = at.i0 - (int64_t)u.p + (int64_t)s * u.d;
                        if (backward) REQUIRE(s >= at.in_lo && s < at.in_hi, "a read of the backward outside the zeros");
                        REQUIRE((s >= at.in_lo && s < at.in_hi) == (x >= -plan.r_front && x < L + plan.r_front), "input row %d of column %d (d %d, p %d)", s, c, u.d, u.p);
                    }
                }
        }
        for (int i = 0; i < u.nout; ++i) REQUIRE(owned[i] == 1, "output %d of kernel %d owned %d times", i, u.k, owned[i]);
    }
}

static void check_split(const PlanHost& plan, int C) {
    for (int mode = 0; mode < 4; ++mode) {
        if (mode == 2 && !resident_backward(plan)) continue;
        for (int N : {1, 2, 3, 7, 24, 100, 149, 1000, 20000, 300000}) {
            const ResidentSplit s = resident_split(plan, N, C, 148, mode);
            REQUIRE(s.examples >= 1 && resident_floats(plan, s.examples, C) <= kRMostFloats, "examples %d", s.examples);
            REQUIRE((int64_t)s.groups * s.examples >= N && (int64_t)(s.groups - 1) * s.examples < N, "groups");
            REQUIRE(s.parts >= 1 && s.parts <= (int)plan.runits.size() && s.run >= 1 && s.run <= s.examples, "parts %d, run %d", s.parts, s.run);
            REQUIRE(s.split == 1 || s.split == 2 || s.split == 4, "split");
            REQUIRE(s.split == 1 || (s.run == 1 && resident_floats(plan, s.examples, C) + resident_merge_floats(plan, s.examples, s.parts, s.split, mode) <= kRMostFloats), "room to merge");
            REQUIRE(s.grid >= 1 && s.grid <= 148 && (int64_t)s.groups * s.parts <= 0x7fffffff, "grid");
        }
    }
}

int main() {
    std::mt19937 rng(5);
    int resident = 0, others = 0, bands[7] = {};
    for (int round = 0; round < 90; ++round) {
        HostParams hp;
        const int Ls[] = {16, 64, 65, 301, 512, 700, 900, 1025, 1100, 1251, 1800, 2047, 2880, 9001};
        const int L = Ls[rng() % 14], C = std::max(1, std::min<int>(255, round % 3 ? (int)(rng() % 40) + 1 : 57600 / L + (int)(rng() % 2)));
        hp.C = C; hp.L = L; hp.K = 40;
        for (int k = 0; k < hp.K; ++k) {
            const int len = (int)(rng() % 3) * 2 + 7, dmax = std::max(1, (L - 1) / (len - 1));
            int d = 1 + (int)(rng() % dmax), p = 0;
            if (k % 3 == 0) d = 1 + (int)(rng() % std::min(dmax, 9));
            if (k % 7 == 0 && round % 2) d = L / 3 + (int)(rng() % L);                            // beyond what random kernels have
            const int span = (len - 1) * d;
            const int lowest = std::max(0, (span - L) / 2 + 1), choices[] = {lowest, std::max(lowest, span / 2), std::max(lowest, (int)(rng() % (span + 3))), std::max(lowest, span + 5)};
            p = choices[round % 2 ? rng() % 4 : rng() % 2];
            const int m = 1 + (int)(rng() % std::min(C, len));
            hp.length.push_back(len); hp.dilation.push_back(d); hp.padding.push_back(p); hp.num_channels.push_back(m);
            hp.bias.push_back(0.5f);
            hp.channel_offset.push_back((int)hp.channel_idx.size());
            hp.weight_offset.push_back((int)hp.weights.size());
            for (int q = 0; q < m; ++q) hp.channel_idx.push_back(q);
            hp.weights.resize(hp.weights.size() + (size_t)m * len, 1.0f);
        }
        hp.channel_offset.push_back((int)hp.channel_idx.size());
        hp.weight_offset.push_back((int)hp.weights.size());
        PlanHost plan;
        build_plan(hp, kSplitDefault, plan, false);
        const bool fits = (int64_t)C * ((L + 3) / 4 * 4) <= kRMostFloats;
        REQUIRE(plan.resident == !plan.runits.empty(), "units for %d x %d", C, L);
        if (!fits || L > kRMostSteps) REQUIRE(!plan.resident, "%d x %d is too long", C, L);
        if (fits && L <= kRMostStepsTested) REQUIRE(plan.resident, "%d x %d fits", C, L);
        ++(plan.resident ? resident : others);
        if (!plan.resident) continue;
        REQUIRE(L <= kRMostStepsTested || plan.r_zeros, "%d steps test their reads", L);
        REQUIRE((int)plan.runits.size() == hp.K, "a kernel is missing");
        {   // the same units where the plan has nothing else
            PlanHost alone;
            build_plan(hp, kSplitDefault, alone, false, true);
            REQUIRE(alone.resident && alone.sitems.empty() == resident_backward(plan), "tiles that no call uses");
            for (int k = 0; k < hp.K; ++k) REQUIRE(alone.krec[alone.runits[k].krec].k == alone.runits[k].k, "record of a unit");
            REQUIRE(alone.flops_s + alone.flops_t > 0.999 * (plan.flops_s + plan.flops_t), "work of a pass");
        }
        check_units(plan, L, false);
        if (resident_backward(plan)) check_units(plan, L, true);
        ++bands[plan.r_bands];
        ++bands[plan.r_back];
        check_split(plan, C);
        REQUIRE(plan.r_pitch >= L + plan.r_front && plan.r_front % 4 == 0 && plan.r_pitch % 4 == 0, "zeros between the rows");
    }
    REQUIRE(resident > 16 && others > 3, "%d handles with units, %d without", resident, others);
    for (int b = 0; b < 7; ++b) REQUIRE(bands[b] > 0, "%d handles with bands %d", bands[b], b);
    std::printf("ok\n");
    return 0;
}
