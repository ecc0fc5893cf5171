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
            CHECK(rows_cluster_size({8, 64, n, 32768}, 148, [](int) { return 0; }) == 0, "nothing fits");
            const int got = rows_cluster_size({8, 3, n, 32768}, 148, [](int c) { return 148 / c; });
            CHECK(got >= 1 && got <= 3, "%d CTAs for 3 key tiles", got);
        }
    std::puts("ok");
    return 0;
}
