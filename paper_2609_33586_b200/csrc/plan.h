// How many CTAs share a work item of the attention forward: cost models fitted to measured times, as plain functions of the
// shape, the SM count and what fits the device, so that they can be tested without one (tests/plan_model.cpp).
#pragma once
#include <algorithm>
#include <cmath>

namespace rowmax {

constexpr int kTileM = 128;  // query rows per tile
constexpr int kTileN = 128;  // keys per tile

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
// and the sum of O; from two thirds of the SMs on they slow each other by a tenth.  512 queries on 16K, 32/8 heads, steady
// streams of calls: bf16 h15 200 -> 164 us, exact 228 -> 148, e4m3 h15 173 -> 119 (2 parts); in streams of 40 calls 64 queries on 8K
// e4m3 90 -> 45 (4 parts).
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
    long long heads;       // (batch, query head) pairs
    int Sq, Sk, D;
    bool causal, exact, fp8;

    int tiles() const { return (Sq + kTileM - 1) / kTileM; }       // query tiles of a head
    int keys(int tile) const {                                     // key tiles that some row of a query tile sees
        const int end = causal ? std::min(Sk, (tile + 1) * kTileM + Sk - Sq) : Sk;
        return end > 0 ? (end + kTileN - 1) / kTileN : 0;
    }
};

// The longest walk of a CTA over items that are dealt as item_index does it: `units` items of each head, the last first, of which
// number u costs cost(u).  Costs fall from the last unit or from the one before it on (a last query tile without a partner), so
// the CTA is one that has the first of these, or one at an end of the row or of the last round.
template <class Cost>
double longest_walk(long long heads, int units, int sms, Cost cost) {
    const long long items = heads * units, ctas = std::min<long long>(items, sms), rounds = (items + ctas - 1) / ctas;
    const auto cta_of = [&](long long w) { return (w / ctas & 1) ? ctas - 1 - w % ctas : w % ctas; };
    const long long likely[4] = {0, ctas - 1, cta_of(items - 1), cta_of(std::min(heads, items - 1))};
    double longest = 0.0;
    for (const long long c : likely) {
        double t = 0.0;
        for (long long r = 0; r < rounds; ++r) {
            const long long w = r * ctas + ((r & 1) ? ctas - 1 - c : c);
            if (w < items) t += cost(units - 1 - static_cast<int>(w / heads));
        }
        longest = std::max(longest, t);
    }
    return longest;
}

// Whether the two-stream form is faster than the plain form, or than the split form where that would give an item `parts` CTAs in
// `split_steps`.  Both walks are added up, in steps of the plain form (a key tile of a pair of query tiles; 0.85 where only one of the
// two sees it): a key tile of one query tile takes 0.52 in the exact modes, 0.58 on fp8 inputs and 0.62 otherwise, an item boundary
// 3.5 against 3.2.  Fitted to 770 measured shapes (2 to 140 key tiles, 1 to 900 query tiles, steady streams of calls): off by 7 %
// (rms).  Times plain -> two streams:
//   A tile for every CTA: as many steps in a row, each of a whole step in the plain form.  16 x 1K e4m3 h15 17.5 -> 14.0 us.
//   Long and short tiles even out: 16 heads x 1408 bf16 h15 22.4 -> 20.5, x 2304 34.9 -> 30.8; not where two rounds are of long tiles
//   alone (2 x 32 heads, 512 queries on 16K 251 -> 301, 4 x 32 heads, 200 on 8K 153 -> 209).
//   Whole rounds: 36 heads x 1337 x 2803 exact, 2 rounds of pairs 92.9, 3 of tiles 83.2; 31 heads, 1123 on 7145 e4m3 h15 150 -> 97.
//   Enough pairs: 48 heads x 2K 61.6 -> 70.3.
// The margins: the plain form keeps calls that the estimate puts within 5 % of each other.  The split form's estimate is low by up to a
// tenth: where it was up to 5 % below the two-stream form's, that took 0.60 to 1.05 times as long.  The exact modes on 16-bit inputs
// stay with it all the same: its parts round P about maxima of their own, so that O would move by 1e-3 (2-norm) with the form and
// lie further from 64-bit results (2.23e-3 -> 2.27e-3, 20 heads, 337 on 2803).  Of the shapes measured the choice of form loses 5 % at
// one and 2 % at another, nowhere else more than 2 %.
// Two or three key tiles: the longer set-up and joining weigh most.  At D = 64 it wins while tiles lie on half of the SMs, so that the
// next call's CTAs can start beside them (2 x 256 6.5 -> 5.7 us, 6 x 380 7.7 -> 7.2; 50 x 148 6.7 -> 7.8), but for a single head of
// three tiles (323 queries 6.75 -> 7.3); beyond that with the exact weights, which gain most (46 x 323 x 193 8.6 -> 7.4), and on
// three key tiles in full attention, where every step of the plain form is a whole one (24 x 711 x 384 9.3 -> 7.9; on two 64 x 256 x
// 256 7.0 -> 7.2).  D = 128 gains or loses a tenth and stays plain.
inline bool streams_pay(const StreamShape& s, int parts, double split_steps, int sms) {
    const int per_head = s.tiles(), nt = (s.Sk + kTileN - 1) / kTileN;
    if (nt < 4) {
        if (s.D != 64 || nt < 2 || (s.heads == 1 && per_head == 3)) return false;
        if (2 * s.heads * per_head > sms && (per_head == 1 || !(s.exact || (nt == 3 && !s.causal)))) return false;
    }
    if (parts > 1 && (per_head == 1 || (s.exact && !s.fp8))) return false;
    const double tile = s.exact ? 0.52 : s.fp8 ? 0.58 : 0.62;
    const double streams = longest_walk(s.heads, per_head, sms, [&](int i) { return s.keys(i) * tile + 3.5; });
    if (parts > 1) return streams < 1.05 * split_steps;
    const double plain = longest_walk(s.heads, (per_head + 1) / 2, sms, [&](int i) {
        const int a = s.keys(2 * i), b = 2 * i + 1 < per_head ? s.keys(2 * i + 1) : 0, both = std::min(a, b);
        return both + 0.85 * (std::max(a, b) - both) + 3.2;
    });
    return 1.05 * streams < plain;
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
// Over the shapes measured the choice costs 0.6 % against always taking the better one, 29 % at most.  (It weighs the plain form alone;
// that the call might otherwise take the two-stream form does not enter.)
inline bool rows_pay(const RowsShape& s, int cs, int sms) { return plain_us(s, sms) >= rows_us(s, cs, sms); }

}  // namespace rowmax
