// Walks the producer of the two-stream form's ring (csrc/kv_ring.cuh: StreamRing) against a model of its mbarriers, of the copies
// and of the MMA warp, which waits for pair G + 2 before the product of tile G and hands a pair back after the scores of its K.
//   stream_ring_model SEEDS      prints the first violation and returns 1, or returns 0
// Looked for: an arrival in a phase whose arrivals have all been made, a wait that lasts for ever, slots overwritten before they
// have been read, and copies that the waits at the end do not cover.
#include "../paper_2609_33586_b200/csrc/kv_ring.cuh"

#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

using rowmax::StreamRing;

namespace {

struct Failure { std::string what; };

struct Barrier {
    int count = 1, pending = 1, tx = 0, phase = 0;
    void init(int n) { count = pending = n; }
    void close() {
        if (pending == 0 && tx == 0) { ++phase; pending = count; }
    }
    void arrive(int bytes, const char* who, int pair) {
        if (pending == 0) throw Failure{std::string("arrival of ") + who + " for pair " + std::to_string(pair) + " in a phase that has all of its arrivals"};
        tx += bytes;
        --pending;
        close();
    }
    bool done(int parity) const { return (phase & 1) != parity; }
};

struct Step { enum { kWait, kScores, kProduct, kRelease } what; int pair; };

template <int NP>
struct World {
    using R = StreamRing<NP>;
    Barrier full[NP], empty[NP];
    int slot[2 * NP];                       // pair whose tile a slot holds, -1 while a copy is under way
    struct Copy { int pair, at; };
    std::vector<Copy> landing;
    std::vector<Step> mma;
    size_t at = 0;
    std::mt19937 rng;
    bool late, gave_up = false;
    int waits_until_abort;

    World(int tiles, unsigned seed, bool late_, int abort_at) : rng(seed), late(late_), waits_until_abort(abort_at) {
        for (auto& b : full) b.init(2);
        for (int& s : slot) s = -1;
        auto scores = [&](int G) { mma.push_back({Step::kScores, G}); mma.push_back({Step::kRelease, G}); };
        for (int G = 0; G < 2 && G < tiles; ++G) { mma.push_back({Step::kWait, G}); scores(G); }
        for (int G = 0; G < tiles; ++G) {
            mma.push_back({Step::kWait, G + 2});
            mma.push_back({Step::kProduct, G + 2});
            if (G + 2 < tiles) scores(G + 2);
        }
    }
    bool land() {
        if (landing.empty()) return false;
        const size_t i = rng() % landing.size();
        const Copy c = landing[i];
        landing.erase(landing.begin() + i);
        slot[c.at] = c.pair;
        Barrier& b = full[R::bar(c.pair)];
        --b.tx;
        b.close();
        return true;
    }
    bool consume() {
        if (at == mma.size()) return false;
        const Step s = mma[at];
        if (s.what == Step::kWait && !full[R::bar(s.pair)].done(R::ph_full(s.pair))) return false;
        if (s.what == Step::kScores && slot[R::slot_k(s.pair)] != s.pair) throw Failure{"scores of pair " + std::to_string(s.pair) + " read another K"};
        if (s.what == Step::kProduct && slot[R::slot_v(s.pair)] != s.pair) throw Failure{"product of pair " + std::to_string(s.pair) + " reads another V"};
        if (s.what == Step::kRelease) empty[R::bar(s.pair)].arrive(0, "the MMA warp", s.pair);
        ++at;
        return true;
    }
    void some() {
        if (!late) for (int n = rng() % 4; n > 0; --n) (rng() & 1) ? land() : consume();
    }
    void arrive(int pair) { some(); full[R::bar(pair)].arrive(0, "the producer", pair); }
    bool wait_empty(int pair) {
        some();
        if (waits_until_abort-- == 0) { gave_up = true; return false; }
        while (!empty[R::bar(pair)].done(R::ph_empty(pair)))
            if (!consume() && !land()) throw Failure{"deadlock at pair " + std::to_string(pair)};
        return true;
    }
    void load(int pair, int to) {
        full[R::bar(pair)].arrive(1, "a load", pair);
        slot[to] = -1;
        landing.push_back({pair, to});
        some();
    }
    void load_k(int pair) { load(pair, R::slot_k(pair)); }
    void load_v(int pair) { load(pair, R::slot_v(pair)); }
};

template <int NP>
void walk(int tiles, unsigned seed, bool late, int abort_at) {
    using R = StreamRing<NP>;
    World<NP> w(tiles, seed, late, abort_at);
    bool ok = true;
    int walked = 0;
    while (ok && walked < tiles)
        if ((ok = rowmax::stream_tile(w, walked))) ++walked;
    int pairs = walked;
    for (int e = walked; ok && e < walked + 2; ++e)
        if ((ok = rowmax::stream_tail(w, e))) pairs = e + 1;
    const int from = pairs > NP ? pairs - NP : 0;
    if (ok) {
        while (w.consume() || w.land()) {}
        if (w.at != w.mma.size() || !w.landing.empty()) throw Failure{"the MMA warp does not get to the end"};
    }
    for (const auto& c : w.landing)
        if (c.pair < from || c.pair >= pairs || !rowmax::stream_pair_is_used(c.pair, walked)) throw Failure{"a copy under way for pair " + std::to_string(c.pair) + " is not waited for at the end"};
    while (w.land()) {}
    for (int pair = from; pair < pairs; ++pair)
        if (rowmax::stream_pair_is_used(pair, walked) && !w.full[R::bar(pair)].done(R::ph_full(pair))) throw Failure{"the wait at the end for pair " + std::to_string(pair) + " runs out"};
}

template <int NP>
void all(int tiles, int seeds) {
    for (int abort_at = -1; abort_at < tiles + 2; ++abort_at)
        for (int s = 0; s <= seeds; ++s) {
            try {
                walk<NP>(tiles, s, s == 0, abort_at);
            } catch (const Failure& f) {
                std::printf("%d pairs, %d tiles, gives up at wait %d, seed %d: %s\n", NP, tiles, abort_at, s, f.what.c_str());
                std::exit(1);
            }
        }
}

}  // namespace

int main(int argc, char** argv) {
    const int seeds = argc > 1 ? std::atoi(argv[1]) : 20;
    for (int tiles = 0; tiles <= 40; ++tiles) {
        all<3>(tiles, seeds);
        all<4>(tiles, seeds);
        all<6>(tiles, seeds);
        all<8>(tiles, seeds);
    }
    std::puts("ok");
    return 0;
}
