// Checks of csrc/plan.h: the plans follow the device that they are made for, and say so when nothing fits it.
#include "../paper_2609_33586_b200/csrc/plan.h"

#include <cstdio>
#include <cstdlib>

using namespace rowmax;

#define CHECK(cond, ...) do { if (!(cond)) { std::printf(__VA_ARGS__); std::printf(": %s\n", #cond); std::exit(1); } } while (0)

int main() {
    // Half a device with half the work plans as the whole one does with all of it.
    const int whole[kMaxSplit + 1] = {0, 148, 74, 46, 36, 28, 24, 20, 18};
    for (int items = 2; items <= 300; items += 2)
        for (int all = 1; all <= 256; all += 1 + all / 7)
            for (int maxima = 0; maxima < 2; ++maxima) {
                const int a = split_parts({static_cast<double>(items), all, all / 3, maxima != 0}, 148, [&](int p) { return whole[p]; });
                const int b = split_parts({items / 2.0, all, all / 3, maxima != 0}, 74, [&](int p) { return whole[p] / 2; });
                CHECK(a >= 1 && a <= kMaxSplit && a <= all, "%d items of %d tiles: %d parts", items, all, a);
                CHECK(items <= 148 || a == 1, "%d items of %d tiles: %d parts", items, all, a);
                CHECK(a == b, "%d items of %d tiles: %d and %d parts", items, all, a, b);
            }
    CHECK(split_parts({4, 128, 128, true}, 148, [](int) { return 0; }) == 1, "nothing fits");
    CHECK(split_parts({4, 128, 128, true}, 148, [&](int p) { return whole[p]; }) > 2, "a few long items");
    for (int cs = 1; cs <= kMaxCluster; ++cs)
        for (int n = 16; n <= 64; n *= 2) {
            CHECK(rows_clusters(n, cs, 0, 148) == 0, "cluster of %d", cs);
            CHECK(rows_clusters(n, cs, 296, 148) == (n == 64 ? 296 : 592), "cluster of %d", cs);
            if (n < 64 && 136 % cs == 0 && cs <= 8) CHECK(rows_clusters(n, cs, 2, 148) == 2 * rows_clusters(n, cs, 1, 74), "cluster of %d", cs);
            CHECK(rows_cluster_size({8, 64, n, 32768, 8, n, 128}, 148, [](int) { return 0; }) == 0, "nothing fits");
            const int got = rows_cluster_size({8, 3, n, 32768, 8, n, 128}, 148, [](int c) { return 148 / c; });
            CHECK(got >= 1 && got <= 3, "%d CTAs for 3 key tiles", got);
        }
    // Measured (us, few-row kernel with that cluster size and plain form): the faster one is taken.
    const struct { RowsShape s; int cs; double rows_us, plain_us; } measured[] = {
        {{32, 1, 16, 32768, 32, 16, 128}, 1, 10.7, 5.2},
        {{4, 1, 16, 16384, 16, 4, 128}, 1, 7.1, 4.4},
        {{64, 1, 16, 8192, 64, 4, 64}, 1, 6.7, 4.6},
        {{2048, 1, 16, 8192, 2048, 11, 64}, 1, 62.6, 48.0},
        {{8, 1, 32, 16384, 8, 32, 128}, 1, 12.7, 4.5},
        {{1, 1, 32, 16384, 8, 24, 64}, 1, 9.3, 4.3},
        {{128, 2, 32, 32768, 128, 24, 128}, 2, 12.4, 7.5},
        {{256, 1, 32, 16384, 256, 24, 128}, 1, 12.9, 9.8},
        {{1024, 1, 64, 32768, 1024, 64, 128}, 1, 173.7, 33.2},
        {{96, 1, 64, 16384, 96, 40, 64}, 1, 14.5, 4.8},
        {{128, 3, 64, 16384, 128, 33, 128}, 1, 19.6, 9.0},
        {{256, 1, 64, 16384, 1024, 44, 128}, 1, 35.9, 27.2},
        {{32, 95, 16, 16384, 256, 8, 128}, 8, 20.4, 228.6},
        {{256, 1, 16, 8192, 1024, 12, 64}, 1, 9.3, 25.2},
        {{512, 10, 16, 16384, 512, 1, 128}, 1, 38.0, 62.6},
        {{8, 6, 16, 16384, 32, 12, 128}, 6, 8.7, 11.3},
        {{256, 30, 32, 8192, 1024, 32, 64}, 1, 66.9, 236.9},
        {{64, 25, 32, 32768, 256, 32, 128}, 4, 28.2, 76.3},
        {{128, 1, 32, 32768, 768, 24, 128}, 1, 12.4, 21.6},
        {{16, 8, 32, 16384, 16, 24, 128}, 8, 10.1, 13.7},
        {{64, 63, 64, 32768, 4096, 64, 128}, 2, 99.9, 2769.4},
        {{4, 35, 64, 16384, 256, 64, 128}, 12, 18.7, 89.9},
        {{16, 2, 64, 16384, 1024, 64, 64}, 2, 14.4, 25.4},
        {{128, 2, 64, 16384, 768, 48, 64}, 1, 16.7, 25.4},
    };
    for (const auto& m : measured)
        CHECK(rows_pay(m.s, m.cs, 148) == (m.rows_us < m.plain_us), "%g groups of %d rows, %d key tiles: %.1f us, plain %.1f us", m.s.groups, m.s.rows, m.s.nt, m.rows_us, m.plain_us);
    // The longest walk, against every CTA's: units of falling cost, the last one as heavy as it is long or a lone tile.
    for (int heads : {1, 3, 16, 18, 31, 36, 74, 148, 155, 400})
        for (int units = 1; units <= 20; ++units)
            for (double last : {1.0, 0.85}) {
                const auto cost = [&](int u) { return (u == units - 1 ? last : 1.0) * (u + 4.0) + 3.0; };
                const int items = heads * units, ctas = std::min(items, 148);
                double longest = 0.0;
                for (int c = 0; c < ctas; ++c) {
                    double t = 0.0;
                    for (int r = 0; r * ctas < items; ++r) {
                        const int w = r * ctas + ((r & 1) ? ctas - 1 - c : c);
                        if (w < items) t += cost(units - 1 - w / heads);
                    }
                    longest = std::max(longest, t);
                }
                const double got = longest_walk(heads, units, 148, cost);
                CHECK(got <= longest && got >= 0.93 * longest, "%d heads of %d units: %g, is %g", heads, units, got, longest);
            }
    // Two streams or what the call would take otherwise (the plain form, or the split form with `parts` CTAs an item), measured in
    // steady streams of calls (us): the faster one is taken.
    const struct { StreamShape s; int parts; double other_us, streams_us; } forms[] = {
        // one tile for every CTA
        {{2, 256, 256, 64, true, false, false}, 1, 6.5, 5.7},
        {{16, 1024, 1024, 128, true, false, true}, 1, 17.5, 14.0},
        {{12, 590, 449, 128, false, false, false}, 1, 15.0, 11.1},
        // two or three key tiles
        {{1, 323, 323, 64, true, false, false}, 1, 6.75, 7.3},
        {{6, 380, 380, 64, true, false, true}, 1, 7.7, 7.2},
        {{46, 323, 193, 64, false, true, false}, 1, 8.6, 7.4},
        {{64, 256, 256, 64, false, false, false}, 1, 7.0, 7.2},
        {{74, 237, 275, 64, true, true, true}, 1, 9.8, 8.3},
        {{24, 711, 384, 64, false, false, true}, 1, 9.3, 7.9},
        {{50, 137, 137, 64, true, false, false}, 1, 6.6, 7.4},
        {{50, 148, 148, 64, true, false, true}, 1, 6.7, 7.8},
        {{37, 274, 274, 64, true, false, true}, 1, 7.7, 8.7},
        {{46, 344, 344, 64, true, false, false}, 1, 8.1, 8.8},
        {{30, 95, 236, 128, true, false, true}, 1, 7.2, 7.4},
        // prompts against themselves, long and short tiles
        {{16, 1408, 1408, 128, true, false, false}, 1, 22.1, 20.5},
        {{16, 1408, 1408, 128, true, true, true}, 1, 21.3, 18.4},
        {{16, 2304, 2304, 128, true, false, false}, 1, 35.3, 31.0},
        {{16, 2048, 2048, 64, true, false, false}, 1, 25.8, 22.5},
        {{32, 1024, 1024, 128, true, false, false}, 1, 19.6, 21.8},
        {{48, 2048, 2048, 128, true, false, false}, 1, 61.6, 70.3},
        {{32, 3001, 3001, 64, true, false, false}, 1, 65.6, 80.1},
        {{16, 8192, 8192, 128, true, true, false}, 1, 272.0, 301.0},
        // chunks on a long context: tiles of nearly one length
        {{64, 512, 16384, 128, true, false, false}, 1, 251.1, 300.5},
        {{64, 512, 16384, 128, true, true, true}, 1, 206.7, 233.9},
        {{32, 1024, 16384, 128, true, false, true}, 1, 180.0, 204.1},
        {{64, 512, 8192, 128, true, true, false}, 1, 152.9, 188.1},
        {{128, 200, 8192, 128, true, false, false}, 1, 153.0, 208.7},
        {{32, 640, 16384, 128, true, false, false}, 1, 203.1, 247.6},
        {{28, 1280, 4000, 64, true, false, false}, 1, 48.3, 54.3},
        {{31, 1123, 7145, 128, true, false, true}, 1, 150.1, 96.6},
        {{25, 1373, 12578, 128, true, true, true}, 1, 290.5, 184.8},
        {{199, 91, 8554, 128, true, true, true}, 1, 184.7, 133.2},
        // full attention: whole rounds
        {{36, 1337, 2803, 128, false, true, false}, 1, 92.9, 83.2},
        {{36, 1337, 2803, 128, false, true, true}, 1, 84.0, 72.4},
        {{32, 8192, 8192, 128, false, true, true}, 1, 816.2, 922.2},
        // the split form
        {{32, 512, 16384, 128, true, false, false}, 2, 163.7, 147.1},
        {{32, 512, 16384, 128, true, false, true}, 2, 118.7, 104.1},
        {{30, 336, 4191, 128, false, false, true}, 2, 43.1, 34.0},
        {{9, 2298, 10402, 64, false, true, false}, 3, 116.4, 141.4},
        {{3, 351, 7263, 128, true, false, false}, 8, 36.9, 58.3},
    };
    for (const auto& f : forms) {
        const int pairs = (f.s.tiles() + 1) / 2, all = f.s.keys(f.s.tiles() - 1), first = std::max(f.s.keys(0), f.s.tiles() > 1 ? f.s.keys(1) : 0);
        for (int part = 1; part <= 2; ++part) {      // the whole device, and half of it with half the heads
            if (f.s.heads % part != 0) continue;
            StreamShape s = f.s;
            s.heads /= part;
            double steps = 0.0;
            const int parts = split_parts({static_cast<double>(s.heads * pairs), all, first, s.fp8 || !s.exact}, 148 / part, [&](int p) { return whole[p] / part; }, &steps);
            CHECK(parts == f.parts, "%lld heads, %d on %d: %d parts", s.heads, s.Sq, s.Sk, parts);
            CHECK(streams_pay(s, parts, steps, 148 / part) == (f.streams_us < f.other_us), "%lld heads, %d on %d, D = %d: %g us in two streams, %g otherwise", s.heads, s.Sq, s.Sk, s.D, f.streams_us, f.other_us);
        }
    }
    // Exact weights on 16-bit inputs: what the split form takes stays with it.
    CHECK(!streams_pay({32, 512, 16384, 128, true, true, false}, 2, 1e6, 148) && streams_pay({32, 512, 16384, 128, true, true, true}, 2, 1e6, 148), "exact weights");
    std::puts("ok");
    return 0;
}
