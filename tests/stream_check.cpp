// Host-side replay of the stream kernel's units (no GPU needed): every output of every kernel it serves is owned exactly once,
// every bulk copy obeys the alignment rules and stays inside the copies, and every word a lane multiplies holds the sample it
// stands for (or a zero outside the series).
#include <cstdio>
#include <vector>

#include "rocket_fast.h"
#include "rocket_fast_geom.h"

using namespace rocket;
using namespace rocket::fast;

namespace rocket { std::atomic<int64_t> g_launch_count{0}; }

#define REQUIRE(cond, ...)                                            \
    do {                                                              \
        if (!(cond)) {                                                \
            std::fprintf(stderr, "FAIL line %d: ", __LINE__);          \
            std::fprintf(stderr, __VA_ARGS__);                        \
            std::fprintf(stderr, "\n");                               \
            return 1;                                                 \
        }                                                             \
    } while (0)

static int check(uint64_t seed, int K, int C, int L, int rows, const HostParams* given = nullptr) {
    HostParams hp;
    if (given) hp = *given;
    else generate_host_params(seed, K, C, L, hp);
    hp.channel_offset.assign(hp.K + 1, 0);
    hp.weight_offset.assign(hp.K + 1, 0);
    for (int k = 0; k < hp.K; ++k) {
        hp.channel_offset[k + 1] = hp.channel_offset[k] + hp.num_channels[k];
        hp.weight_offset[k + 1] = hp.weight_offset[k] + hp.num_channels[k] * hp.length[k];
    }
    PlanHost plan;
    build_plan(hp, kSplitDefault, plan);
    REQUIRE(plan.wunits.empty() == plan.titems.empty(), "units for the kernels of the large dilations");
    std::vector<std::vector<uint8_t>> cover(plan.krec.size());
    for (size_t f = 0; f < plan.krec.size(); ++f) cover[f].assign(plan.krec[f].nout, 0);
    const int64_t pitch = plan.wpitch, front = plan.wfront, copies = (int64_t)rows * kWCopies;
    const int64_t room = copies * pitch + front + pitch;         // what ensure_stream_capacity allocates
    REQUIRE(pitch % 4 == 0 && front % 4 == 0 && pitch >= L + front, "pitch");
    for (const WUnit& u : plan.wunits) {
        const KRec& f = plan.krec[u.krec];
        const int R = u.shape & 0xff, len = (u.shape >> 8) & 0xff, row_xor = u.shape >> 16, G = w_rows_per_y(u.d), S = R + len - 1;
        const WMapSpec& sp = plan.wmaps.at(u.map);
        REQUIRE(f.d == u.d && f.len == len && f.m == u.m && f.k == u.k && f.p == u.p && f.lo_u == u.lo_u && f.hi_u == u.hi_u && f.tl == u.tl &&
                f.rl == u.rl && f.th == u.th && f.rh == u.rh && f.nout == u.nout && f.woff == u.woff && f.d >= plan.split, "unit fields");
        REQUIRE((R == 16 || R == 12 || R == 8) && u.ntiles >= 1 && u.ncol == (u.d + 63) / 64 && u.run == G * u.d && u.band_y == R / G, "unit shape");
        REQUIRE(sp.d == u.d && sp.y_rows * G >= S && u.bytes == sp.y_rows * G * kWarpCols * 4 && u.bytes <= kWStageFloats * 4, "box");
        for (int q = 0; q < u.m; ++q) REQUIRE(u.ch[q] == f.ch[q] && u.ch[q] < hp.C, "channels");
        // the tensor map, as ensure_stream_capacity encodes it
        const int64_t d = u.d, run = u.run;
        const int64_t step = d % 4 == 1 ? pitch + d - 1 : d % 4 == 3 ? pitch - d - 1 : d % 4 == 2 ? 2 * pitch + d - 2 : pitch;
        const int64_t ny = (front + L + (d % 4 == 3 ? 3 * d : 0) + run - 1) / run;
        REQUIRE(step % 4 == 0 && step > 0 && run % 4 == 0, "strides are multiples of 16 bytes");
        for (int t = u.tile0; t < u.tile0 + u.ntiles; ++t) {
            const int band = t / u.ncol, c0 = 64 * (t % u.ncol), trow = u.t0 + band * R;
            int64_t x = u.x0 + c0, y = u.y0 + (int64_t)band * u.band_y;
            while (x >= run) { x -= run; ++y; }
            REQUIRE(x % 4 == 0 && x >= 0 && x + kWarpCols <= run + kWarpCols, "box x");
            for (int64_t rho : {(int64_t)0, (int64_t)rows - 1})   // first and last channel row
                for (int s = 0; s < S; ++s) {
                    const int stage_row = (s >> 2 << 2) + ((s & 3) ^ row_xor), yy = stage_row / G, i = stage_row % G;
                    REQUIRE(stage_row < sp.y_rows * G, "row outside the box");
                    for (int c : {0, 1, 62, 63}) {
                        const int64_t want = (int64_t)(trow + s) * d + c0 + c;        // sample index
                        const bool filled = y + yy < 0 || y + yy >= ny;
                        if (filled) { REQUIRE(want < 0 || want >= L, "zero fill where a sample is expected"); continue; }
                        const int64_t at = (rho * kWCopies + u.copy) * pitch + (y + yy) * run + i * step + x + c;
                        REQUIRE(at >= 0 && at < room, "read outside the copies");
                        const int64_t cp = u.copy + (d % 4 == 1 ? i : d % 4 == 3 ? i : d % 4 == 2 ? 2 * i : 0);
                        REQUIRE(cp >= 0 && cp < kWCopies, "no such copy");
                        // copy cp holds the layout moved down by cp floats
                        const int64_t layout = at - (rho * kWCopies + cp) * pitch + cp;
                        REQUIRE(layout == front + want, "wrong sample: kernel %d (d %d len %d) row %d: got %lld, want %lld", u.k, u.d, len, s,
                                (long long)(layout - front), (long long)want);
                        // positions without a sample lie in the zeros between two copies
                        if (want < 0 || want >= L)
                            REQUIRE(layout - cp >= front - pitch + L && layout - cp < pitch + front - kWCopies, "reads a neighbouring copy's samples");
                    }
                    // rows of the box beyond the tile's need stay inside the room as well
                }
            const int64_t far = ((int64_t)(rows - 1) * kWCopies + u.copy) * pitch + (ny - 1) * run + (G - 1) * step + run + kWarpCols;
            REQUIRE(far <= room, "box beyond the allocation");
            for (int o = 0; o < R; ++o)
                for (int c = 0; c < 64; ++c) {
                    const int64_t v = (int64_t)(trow + o) * d + c0 + c;
                    if (c0 + c < d && v >= u.lo_u && v < u.hi_u) cover[u.krec][v + u.p]++;
                }
        }
    }
    for (size_t f = 0; f < plan.krec.size(); ++f)
        for (int i = 0; i < plan.krec[f].nout; ++i)
            REQUIRE(cover[f][i] == (plan.krec[f].d >= plan.split && !plan.wunits.empty() ? 1 : 0), "kernel %d (len %d d %d p %d) output %d owned %d times",
                    plan.krec[f].k, plan.krec[f].len, plan.krec[f].d, plan.krec[f].p, i, (int)cover[f][i]);
    std::printf("ok L=%d: %zu units, %zu maps\n", L, plan.wunits.size(), plan.wmaps.size());
    return 0;
}

int main() {
    int rc = 0;
    rc |= check(8527, 1500, 20, 5000, 40);
    rc |= check(11, 400, 20, 50000, 40);
    rc |= check(12, 400, 7, 10001, 84);
    rc |= check(13, 300, 3, 997, 3);
    rc |= check(21, 150, 20, 200000, 20);
    // paddings that are no multiples of the dilation, beyond the usual, and the largest dilations
    HostParams hp;
    hp.K = 0; hp.C = 2; hp.L = 1000;
    auto add = [&](int len, int d, int p) {
        hp.length.push_back(len); hp.dilation.push_back(d); hp.padding.push_back(p); hp.num_channels.push_back(1);
        hp.channel_idx.push_back(1); hp.bias.push_back(0.5f);
        for (int j = 0; j < len; ++j) hp.weights.push_back(1.0f);
        hp.K++;
    };
    add(7, 166, 0); add(7, 166, 498); add(11, 99, 495); add(7, 64, 5); add(9, 65, 300); add(11, 100, 1); add(7, 127, 381);
    add(7, 128, 0); add(9, 124, 0); add(7, 129, 5); add(9, 77, 308); add(11, 91, 2); add(7, 131, 900); add(9, 130, 2000);
    add(7, 330, 990); add(7, 340, 1000); add(7, 512, 1536); add(11, 345, 1725); add(7, 67, 1); add(9, 66, 263);
    rc |= check(0, hp.K, hp.C, hp.L, 2, &hp);
    return rc;
}
