// How many CTAs share a work item of the attention forward: cost models fitted to measured times, as plain functions of the
// shape, the SM count and what fits the device, so that they can be tested without one (tests/plan_model.cpp).
#pragma once
#include <algorithm>
#include <cmath>

namespace rowmax {

constexpr int kMaxSplit = 8;     // CTAs that share an item in the split form (the portable cluster size)
constexpr int kMaxCluster = 16;  // CTAs that share a (batch, key/value head) in the few-row kernel

// The machine that the figures were measured on.  Counts of SMs below are shares of it.
constexpr int kMeasuredSms = 148;

struct SplitShape {
    double items;       // pairs of query tiles of all (batch, head)
    int all, first;     // key tiles of the longest pair and of the first one
    bool takes_maxima;  // the parts need the row maxima of the parts before them
};

// CTAs per item, 1 for the plain form.  fit(parts): clusters of that size that fit the device at once.  Times are in steps of the
// loop (one key tile of a pair of query tiles), measured: a part costs its key tiles, with a maxima pass 0.65 of a step more for
// each tile of its maxima pass (two parts share the pass, so it is half as long), and 4.5 steps + 0.5 per part for the exchange
// and the sum of O; from two thirds of the SMs on they slow each other by a tenth.  512 queries on 16K, 32/8 heads, streams of 40
// calls: bf16 h15 218 -> 143 us, exact 256 -> 134, e4m3 h15 203 -> 132 (2 parts); 64 queries on 8K e4m3 90 -> 45 (4 parts).
// 16 x 1K and 16 x 2K gain nothing and stay whole.
// *steps gets the estimated time.
template <class Fit>
int split_parts(const SplitShape& s, int sms, Fit fit, double* steps = nullptr) {
    if (s.items > sms) return 1;
    const double longest = s.all, mean = 0.5 * (s.all + s.first);
    double best = 0.93 * (longest + 1.5);      // a gain below that is not worth the risk of being wrong
    int best_parts = 1;
    for (int parts = 2; parts <= kMaxSplit && parts <= s.all; ++parts) {
        const int n = fit(parts);
        if (n <= 0) continue;
        const double per_tile = (!s.takes_maxima ? 1.0 : parts == 2 ? 1.325 : 1.65) / parts;
        const double fixed = 4.5 + 0.5 * parts, busy = s.items * parts * kMeasuredSms > 100.0 * sms ? 1.1 : 1.0;
        const double waves = std::ceil(s.items / n);
        const double t = std::fmax(longest * per_tile + fixed, waves * (mean * per_tile + fixed)) * busy;
        if (t < best) { best = t; best_parts = parts; }
    }
    if (steps != nullptr) *steps = best;
    return best_parts;
}

struct StreamShape {
    double tiles, pairs;   // query tiles, and pairs of them, of all (batch, head)
    int per_head;          // query tiles of a head
    int nt;                // key tiles of the longest
    int D;
    bool causal;
    bool one_anchor;       // all but the exact modes on 16-bit inputs
};

// Whether the two-stream form (one query tile per CTA) is faster than the plain form, or than the split form where that would
// give an item `parts` CTAs in `split_steps`.  In steps of the plain form, measured over 60 shapes: a key tile of one query tile
// takes 0.64 (0.56 in the exact modes on 16-bit inputs), an item boundary 3.0 against the plain form's 3.6.
//   One tile per CTA: the plain form has as many steps in a row, each of a whole step.  Lost only to the longer set-up and joining of
//   a few key tiles (D = 128: 3 tiles 8.9 -> 9.4 us, 5 to 12 tiles 21.9 -> 15.9 and 22.7 -> 16.2; D = 64: 2 tiles 8.3 -> 6.1).
//   Causal, one pair but more than one tile per CTA: long and short tiles even out over two rounds (16 heads x 1408 23.8 -> 19.6 us,
//   x 2304 36.2 -> 31.3), from 12 key tiles on (8 tiles 32.9 -> 40.1, which have three rounds).
//   Full attention, all items equal: whole rounds decide (36 heads x 1337 x 2803 exact: 2 rounds of pairs 94 us, 3 of tiles 76).
//   Other shapes have enough pairs: 48 heads x 2K 57.8 us in the plain form, 68.2 in this one.
inline bool streams_pay(const StreamShape& s, int parts, double split_steps, int sms) {
    const double tile = s.one_anchor ? 0.64 : 0.56, boundary = 3.0;
    if (s.nt < (s.D == 64 ? 2 : 4)) return false;
    if (parts > 1) return s.per_head > 1 && s.tiles <= sms && s.nt * tile + boundary < split_steps;
    if (s.tiles <= sms) return true;
    if (s.causal) return s.pairs <= sms && s.tiles <= 2.0 * sms && s.nt >= 12;
    return 1.08 * std::ceil(s.tiles / sms) * (s.nt * tile + boundary) < std::ceil(s.pairs / sms) * (s.nt + 3.6);
}

struct RowsShape {
    double groups;      // (batch, key/value head) pairs
    int nt;             // key tiles
    int n;              // rows of the tile: 16, 32 or 64
    int tile_bytes;     // of K or V
    double items;       // (batch, query head) pairs: the plain form's work items
    int rows, D;        // rows that the tile holds, head dimension
};

// Clusters of cs CTAs that the few-row kernel can have on the device, given what the occupancy query says.  The query counts one
// CTA per SM for every kernel that allocates TMEM; tiles of 16 and 32 rows run two, and a cluster may then lie on half as many
// SMs, so that of the portable sizes 272 of the 2 x 148 places can be used.
inline int rows_clusters(int n_rows, int cs, int queried, int sms) {
    if (n_rows == 64 || queried <= 0) return queried;
    return cs <= 8 ? std::max(272 * sms / kMeasuredSms / cs, 2 * queried) : 2 * queried;
}

// CTAs per cluster of the few-row kernel, 0 if none fits: the candidate with the shortest estimated time.  Measured on shapes
// from 1 x 1K to 16 x 2K and 1 x 32K: a part that does not depend on the context (5.6 us, 0.1 us per CTA of a cluster for exchange
// and combination, 1.2 us more beyond the portable size), one key tile's way through a CTA (hand-offs 0.83 us, or the rate of
// 55 GB/s one CTA reads at), and the device's bandwidth, which are added as squares where they overlap.  It picks the fastest
// size or one within 8 % of it.  fit(cs): what the occupancy query says.
template <class Fit>
int rows_cluster_size(const RowsShape& s, int sms, Fit fit) {
    const double bytes_us = 2.0 * s.nt * s.groups * s.tile_bytes / 6.3e6;
    const double pair_us = std::fmax(s.n == 16 ? 0.83 : s.n == 32 ? 1.6 : 2.5, 2.0 * s.tile_bytes / 55e3);
    double best = 1e30;
    int best_cs = 0;
    for (int cs = 1; cs <= kMaxCluster && cs <= s.nt; ++cs) {
        const int n = rows_clusters(s.n, cs, fit(cs), sms);
        if (n <= 0) continue;
        const double waves = std::ceil(s.groups / n);
        const double shared = std::fmin(s.groups, n) * cs > sms ? 1.15 : 1.0;     // two CTAs on an SM slow each other a little
        const double hand_us = waves * ((s.nt + cs - 1) / cs) * pair_us * shared;
        const double t = waves * (5.6 + 0.1 * cs + (cs > 8 ? 1.2 : 0.0)) + std::sqrt(hand_us * hand_us + bytes_us * bytes_us);
        if (t < best) { best = t; best_cs = cs; }
    }
    return best_cs;
}

// Estimated times (us) of the two kernels that a forward with few rows can take, fitted to 700 measured shapes (1 to 64 rows, 1 to
// 140 key tiles, 1 to 4096 heads; graph replays): off by 8 % (rms).  The kernels' own work and the reading of K and V overlap and
// are added as squares.
inline double rows_us(const RowsShape& s, int cs, int sms) {
    struct Fit { double fixed, per_row, per_tile, per_cta, start, rate; };
    const Fit f = s.n == 16 ? Fit{5.35, 0.286, 0.699, 0.213, 1.93, 0.927} :
                  s.n == 32 ? Fit{5.42, 0.181, 1.393, 0.150, 3.88, 1.118} : Fit{7.05, 0.197, 2.146, 0.161, 6.32, 0.876};
    const double read_us = f.start + f.rate * 2.0 * s.nt * s.groups * s.tile_bytes / 6.3e6;
    const double places = s.n == 64 ? sms : 2.0 * sms, waves = std::ceil(s.groups * cs / places);
    const double shared = std::fmin(s.groups, std::floor(places / cs)) * cs > sms ? 1.15 : 1.0;
    const double work_us = waves * (f.fixed + f.per_row * s.rows * s.D / 128.0 / cs + f.per_cta * cs + (cs > 8 ? 1.2 : 0.0) +
                                    (s.nt + cs - 1) / cs * f.per_tile * shared);
    return std::sqrt(work_us * work_us + read_us * read_us);
}
inline double plain_us(const RowsShape& s, int sms) {      // one pair of query tiles per head: at most 64 rows
    const double rounds = std::ceil(s.items / sms), read_us = 1.49 + 2.0 * s.nt * s.groups * s.tile_bytes / 6.3e6;
    const double work_us = 1.85 + rounds * (1.83 + s.nt * (s.D == 64 ? 1.05 : 1.30)) + (rounds > 1.0 ? 1.41 : 0.0);
    return std::sqrt(work_us * work_us + read_us * read_us);
}
// Whether the few-row kernel with clusters of cs CTAs is the faster one.  Its epilogue costs 0.18 to 0.29 us for each row of a
// CTA, which many short heads do not earn back: 1024 heads x 64 rows x 1 key tile 174 us against 33 in the plain form, 32 x 48
// rows x 1 tile 18.2 against 4.8.  It wins once the keys are read for long enough: 32 groups of 8 rows x 95 tiles 20 against 229.
// Over the shapes measured the choice costs 0.6 % against always taking the better one, 29 % at most.
inline bool rows_pay(const RowsShape& s, int cs, int sms) { return plain_us(s, sms) >= rows_us(s, cs, sms); }

}  // namespace rowmax
