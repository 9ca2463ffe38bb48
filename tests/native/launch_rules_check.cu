// Host-side check of the rules that choose a call's launch shape (no GPU needed): a rule leaves no SM
// idle that the work could use, and stays within the buffers the plan has.
// Usage: launch_rules_check   (exit status 0 when every check holds)
#include <algorithm>
#include <cstdio>

#include "epic_internal.cuh"

static long g_bad = 0;
#define CHECK(cond, ...)                  \
    do {                                  \
        if (!(cond)) {                    \
            if (g_bad < 20) {             \
                std::printf(__VA_ARGS__); \
                std::printf("\n");        \
            }                             \
            g_bad++;                      \
        }                                 \
    } while (0)

// Image series in the compact kernel: one CTA per channel and time chunk, so a batch of few images
// splits each, within the partial images of the plan.
static void series()
{
    for (int sms : {148, 152})
        for (int chan : {1, 3, 12, 32, 64, 200})
            for (int img : {1, 2, 3, 10, 25})
                for (int spi : {1, 8, 40, 100, 1000})
                    for (int cap : {img, 2 * img + 1, 64}) {
                        const int n = epic::series_chunks(chan, img, spi, cap, sms);
                        CHECK(n >= 1 && n * img <= std::max(cap, img) && n <= spi, "%d chunks of %d x %d spectra, cap %d", n, img,
                              spi, cap);
                        // the batch's time, in samples on the busiest SM (4 for set-up and partial image)
                        auto cost = [&](int k) { return ((chan * img * k + sms - 1) / sms) * ((spi + k - 1) / k + 4.0); };
                        for (int k = 1; k * img <= cap && k <= spi; k++)
                            CHECK(cost(n) <= cost(k) + 1e-9, "%d channels, %d x %d spectra: %d chunks cost %g, %d cost %g", chan,
                                  img, spi, n, cost(n), k, cost(k));
                    }
}

// Side 64: images per class where the gather is small (the measured pairs beside the rule).
static void side64()
{
    const struct {
        int P, A, K, span;
        bool compact;
    } at[] = {{1, 64, 5, 56, false}, {1, 64, 7, 56, false}, {1, 64, 3, 15, false}, {1, 32, 5, 15, false}, {1, 64, 5, 16, true},
              {1, 256, 3, 15, true},  {2, 16, 1, 14, false}, {2, 16, 1, 56, false}, {2, 32, 3, 15, true},  {2, 256, 5, 40, true}};
    CHECK(!epic::compact_pays_odd(64, 1, 1) && epic::compact_pays_odd(64, 1, 3) && epic::compact_pays_odd(64, 2, 1) &&
              epic::compact_pays_odd(96, 1, 1), "odd rows");
    for (const auto &c : at) {
        CHECK(epic::compact_pays(64, c.P, c.A, c.K, c.span, c.span) == c.compact, "side 64, P %d, %d antennas, K %d, %d cells", c.P,
              c.A, c.K, c.span);
        for (int N : {96, 128}) CHECK(epic::compact_pays(N, c.P, c.A, c.K, c.span, c.span), "side %d", N);
    }
}

// Epilogue: one pixel a thread only where four would leave SMs without a block (measured pairs).
static void tiles()
{
    const struct {
        int N, images, want;
    } at[] = {{32, 4, 4}, {128, 4, 64}, {128, 16, 16}, {128, 32, 16}, {64, 32, 16}, {64, 64, 4}, {64, 150, 4}, {512, 1, 256}, {128, 8, 64}};
    for (const auto &c : at)
        CHECK(epic::epi_tiles(c.N, 2, c.images, 152) == c.want, "side %d, %d images: %d tiles", c.N, c.images,
              epic::epi_tiles(c.N, 2, c.images, 152));
    CHECK(epic::epi_tiles(128, 1, 10, 152) == 64 && epic::epi_tiles(64, 1, 38, 152) == 16 && epic::epi_tiles(128, 1, 16, 152) == 16,
          "one polarisation");
}

// Side 32 alone: no fork beside one wave of long chunks (measured pairs).
static void fork32()
{
    CHECK(!epic::fork_pays(152, 1, 500, 152, 2, 2304) && !epic::fork_pays(152, 1, 500, 152, 2, 144), "one long wave");
    CHECK(epic::fork_pays(4, 32, 64, 152, 1, 144) && epic::fork_pays(64, 7, 200, 152, 2, 144) && epic::fork_pays(20, 7, 81, 152, 1, 3726),
          "short wave, several waves");
}

// E-field calls: per class while its CTAs fit on the SMs at once (measured pairs).
static void efield()
{
    const struct {
        int N, P, items, T;
        bool classes;
    } at[] = {{128, 2, 16, 8, true}, {128, 2, 16, 12, true}, {128, 2, 32, 8, true}, {128, 2, 20, 14, true},  {128, 2, 16, 20, false}, {128, 2, 256, 1, false},
              {128, 1, 16, 8, true}, {128, 1, 64, 8, true},  {128, 1, 256, 2, false}, {96, 2, 16, 12, true}, {96, 2, 16, 20, false},
              {64, 2, 4, 1, false}};
    for (const auto &c : at)
        CHECK(epic::efield_per_class(c.N, c.P, c.items, c.T, 152) == c.classes, "side %d, P %d, %d classes x %d spectra", c.N, c.P,
              c.items, c.T);
}

// Wide kernels: buffers within their budgets, no FP32 sum longer than the per-class kernel's (side 256), and
// long calls as well spread over the SMs as short ones.
static void wide()
{
    const int sms = 152;
    for (int N : {256, 512})
        for (int chan : {1, 2, 16, 63, 64, 256, 1000})
            for (int rpad : {32, 128})
                for (int most : {1, 7, 100, 500, 1000, 5000, 9000, 20000}) {
                    const int Q = N / 64, items = chan * Q * Q, tau = epic::fp32_pick_tau(items, most, sms);
                    const epic::WideLayout w = epic::wide_layout(N, chan, rpad, most, 0, tau, sms);
                    const double work = static_cast<double>(w.cb) * w.tb * N * 2 * rpad * 8;
                    CHECK(w.cb >= 1 && w.cb <= chan && w.tb >= 1 && work <= 4.0 * (1ull << 30), "workspace: %d x %d", w.cb, w.tb);
                    const double slot = static_cast<double>(chan) * N * N * 16;
                    CHECK(w.slots <= tau || w.slots * slot <= 2.0 * (1ull << 30), "%d partial images of %g bytes", w.slots, slot);
                    for (int T : {1, 2, 50, most / 2, most - 1, most}) {
                        if (T < 1 || T > most) continue;
                        const epic::WideSplit s = epic::wide_split(N, items, w.cb, w.tb, w.slots, T, sms);
                        const int nb = (T + s.batches - 1) / s.batches, n = (nb + s.n_sub - 1) / s.n_sub;
                        CHECK(s.batches % s.rounds == 0 && s.n_sub * s.rounds <= w.slots && nb <= w.tb, "side %d, %d channels, %d of %d: "
                              "%d batches, %d x %d of %d slots", N, chan, T, most, s.batches, s.n_sub, s.rounds, w.slots);
                        const int per_class = std::min(tau, epic::fp32_pick_tau(items, T, sms)), per_slot = s.batches / s.rounds;
                        if (N == 256)
                            CHECK(per_slot * n <= (T + per_class - 1) / per_class + 2 * per_slot, "side %d, %d channels, %d spectra: sums of %d",
                                  N, chan, T, per_slot * n);
                        // samples of column work on the busiest SM against an even spread
                        if (T != most || T < 500) continue;
                        double busy = 0;
                        for (int c0 = 0; c0 < chan; c0 += w.cb) {
                            const long long blocks = static_cast<long long>(std::min(w.cb, chan - c0)) * 2 * Q * s.n_sub;
                            busy += static_cast<double>(s.batches) * ((blocks + sms - 1) / sms) * n;
                        }
                        const double even = std::max(1.0 * T * chan * 2 * Q / sms, T / 64.0);
                        CHECK(busy <= 1.25 * even, "side %d, %d channels, %d rows, %d spectra: %g samples, %g if even", N, chan, rpad, T, busy,
                              even);
                    }
                }
}

// The shapes by which test_gpu_wide.py continues sums in a partial image and images channels in two groups
static void wide_test_shapes()
{
    const struct {
        int N, C, T, most, cap, rpad;
        bool more;      // batches beyond the first set of partial images
        int groups;
    } at[] = {{512, 2, 7, 7, 1, 112, true, 1}, {512, 2, 7, 7, 3, 112, true, 1},   {256, 2, 16, 16, 1, 128, true, 1},
              {256, 2, 8, 8, 3, 128, false, 1}, {512, 63, 2, 100, 200, 128, false, 2}, {512, 9, 5, 5, 2, 80, true, 1}};
    for (const auto &c : at) {
        const int items = c.C * (c.N / 64) * (c.N / 64);
        const epic::WideLayout w = epic::wide_layout(c.N, c.C, c.rpad, c.most, c.cap, epic::fp32_pick_tau(items, c.most, 152), 152);
        const epic::WideSplit s = epic::wide_split(c.N, items, w.cb, w.tb, w.slots, c.T, 152);
        CHECK((s.batches > s.rounds) == c.more && (c.C + w.cb - 1) / w.cb == c.groups, "side %d, %d x %d: %d batches, %d rounds, %d channels",
              c.N, c.C, c.T, s.batches, s.rounds, w.cb);
    }
}

// A stage of two groups: the time either ran, not the span between them
static void stage_time()
{
    CHECK(epic::stage_union(0, 2, 10, 13) == 5 && epic::stage_union(0, 2, -7, -4) == 5, "apart");
    CHECK(epic::stage_union(0, 4, 3, 9) == 9 && epic::stage_union(0, 9, 2, 5) == 9 && epic::stage_union(0, 3, -2, 1) == 5, "overlapping");
}

// A wide group's small calls go to the per-class kernel, whose time chunks are tuned like any other's
static void tuning()
{
    epic_plan_s plan;
    plan.A = 300;
    plan.K = 5;
    epic::GroupCfg g;
    g.N = 256;
    g.n_items = 2 * 16;
    CHECK(epic::tunable(&plan, g, 16), "per-class group");
    g.wide = true;
    CHECK(epic::tunable(&plan, g, 16) && !epic::tunable(&plan, g, 100), "wide group, small and ordinary call");
    g.wide = false;
    g.alias = true;
    CHECK(!epic::tunable(&plan, g, 16), "fold path");
}

static void efield_plans()
{
    CHECK(epic::efield_tables(128, 2, 16, 1000, 152) && epic::efield_tables(128, 2, 32, 8, 152), "few channels, short calls");
    CHECK(!epic::efield_tables(128, 2, 32, 1000, 152) && !epic::efield_tables(64, 2, 4, 1, 152), "more channels, long calls; side 64");
}

// Gain solver: clusters where they are the faster form (measured pairs), in one wave where that is possible
static void gains()
{
    const struct {
        int A, P, C, T;
        bool cluster;
    } at[] = {{256, 2, 61, 8, false}, {256, 2, 61, 20, false}, {256, 2, 61, 66, true},    {256, 2, 64, 1000, true}, {34, 1, 8, 20, false},
              {512, 2, 8, 20, false}, {512, 2, 200, 66, false}, {512, 2, 200, 200, true}, {297, 2, 200, 1000, false},
              {600, 1, 8, 8, false},  {600, 1, 8, 20, true},   {1001, 1, 200, 200, true}, {297, 2, 61, 66, false},    {513, 2, 4, 1000, false}};
    for (const auto &c : at)
        CHECK((epic::cal_cluster_size(c.A * c.P, c.P, c.C, c.T, 152) > 0) == c.cluster, "%d x %d, %d channels, %d spectra", c.A, c.P, c.C,
              c.T);
    for (int AP : {64, 512, 600, 1024})
        for (int C : {1, 19, 38, 61, 64, 76, 77, 152, 153, 304})
            for (int T : {64, 128, 1000}) {
                const int cl = epic::cal_cluster_size(AP, 2, C, T, 152), room = AP > 512 ? 152 : 304;
                CHECK(cl <= 1 || cl * C <= room, "%d values, %d channels: clusters of %d", AP, C, cl);
            }
}

int main()
{
    gains();
    efield_plans();
    tuning();
    stage_time();
    wide();
    wide_test_shapes();
    efield();
    fork32();
    tiles();
    side64();
    series();
    if (g_bad) std::printf("%ld checks failed\n", g_bad);
    return g_bad ? 1 : 0;
}
