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
    // Two streams or the plain form, measured (us): the faster one is taken.
    const struct { StreamShape s; bool streams; } forms[] = {
        {{4, 2, 2, 2, 64, true, true}, true},            // 8.3 against 6.1
        {{128, 64, 8, 8, 128, true, true}, true},        // 17.7, 14.1
        {{396, 216, 11, 22, 128, false, false}, true},   // 94, 76
        {{396, 216, 11, 22, 128, false, true}, false},
        {{288, 144, 18, 18, 128, true, true}, true},     // 36.2, 31.3
        {{768, 384, 16, 16, 128, true, true}, false},    // 57.8, 68.2
        {{768, 384, 24, 24, 64, true, true}, false},     // 66.2, 79.9
        {{48, 32, 3, 3, 128, true, false}, false},       // 8.9, 9.4
        {{280, 144, 35, 35, 128, false, true}, false},   // 61.3, 72.6
    };
    for (const auto& f : forms) CHECK(streams_pay(f.s, 1, 0.0, 148) == f.streams, "%g query tiles, %d key tiles", f.s.tiles, f.s.nt);
    std::puts("ok");
    return 0;
}
