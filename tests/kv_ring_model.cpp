// Walks the producer of csrc/kv_ring.cuh against a model of its mbarriers, of the copies and of the MMA warp.
//   kv_ring_model SEEDS      prints the first violation and returns 1, or returns 0
// A barrier is a pending count and a byte count; a phase ends when both are zero.  The violation looked for is an arrival in a
// phase whose arrivals have all been made (its bytes still under way): undefined for an mbarrier.  Copies land in any order:
// "late" lets nothing land and nobody read until the producer cannot go on, the others mix the steps at random.
#include "../paper_2609_33586_b200/csrc/kv_ring.cuh"

#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

using rowmax::KvRing;

namespace {

struct Failure { std::string what; };

struct Barrier {
    int count = 1, pending = 1, tx = 0, phase = 0;
    void init(int n) { count = pending = n; }
    void close() {
        if (pending == 0 && tx == 0) { ++phase; pending = count; }
    }
    void arrive(int bytes, const char* who, int idx) {
        if (pending == 0) throw Failure{std::string("arrival of ") + who + " at position " + std::to_string(idx) + " in a phase that has all of its arrivals"};
        tx += bytes;
        --pending;
        close();
    }
    bool done(int parity) const { return (phase & 1) != parity; }     // the phase of that parity has ended
};

struct Item { int pre, n; };
struct Step { bool wait; int idx; };      // of the MMA warp: wait for a full barrier, or commit to an empty one

template <int NS>
struct World {
    using R = KvRing<NS>;
    Barrier full[R::kPairs], empty[R::kPairs];
    std::vector<Step> mma;
    std::vector<int> landing;         // positions whose copies are under way
    size_t at = 0;
    std::mt19937 rng;
    bool late, abort_now = false;
    int waits_until_abort;            // the producer gives up at this wait (< 0: never)

    World(const std::vector<Item>& items, unsigned seed, bool late_, int abort_at) : rng(seed), late(late_), waits_until_abort(abort_at) {
        for (auto& b : full) b.init(2);
        int base = 0;
        for (const Item& it : items) {
            for (int j = 0; j < it.pre; ++j, ++base) {
                if (base == 0 || (base & 1)) mma.push_back({true, base});
                if ((base & 1) == 0) mma.push_back({false, base});
            }
            base += base & 1;
            if (it.n > 0) {
                mma.push_back({true, base});
                mma.push_back({false, base});
                for (int j = 0; j < it.n; ++j) {
                    mma.push_back({true, base + 2 * j + 1});
                    if (j + 1 < it.n) mma.push_back({false, base + 2 * j + 2});
                }
            }
            base += 2 * it.n;
        }
    }
    bool land() {
        if (landing.empty()) return false;
        const size_t i = rng() % landing.size();
        Barrier& b = full[R::bar(landing[i])];
        --b.tx;
        b.close();
        landing.erase(landing.begin() + i);
        return true;
    }
    bool consume() {
        if (at == mma.size()) return false;
        const Step s = mma[at];
        if (s.wait && !full[R::bar(s.idx)].done(R::ph_full(s.idx))) return false;
        if (!s.wait) empty[R::bar(s.idx)].arrive(0, "the MMA warp", s.idx);
        ++at;
        return true;
    }
    void some() {      // between the producer's steps
        if (!late) for (int n = rng() % 4; n > 0; --n) (rng() & 1) ? land() : consume();
    }
    // ---- what the producer calls
    void arrive(int idx) { some(); full[R::bar(idx)].arrive(0, "the producer", idx); }
    bool wait_empty(int idx) {
        some();
        if (abort_now || waits_until_abort-- == 0) { abort_now = true; return false; }
        while (!empty[R::bar(idx)].done(R::ph_empty(idx)))
            if (!consume() && !land()) throw Failure{"deadlock at position " + std::to_string(idx)};
        return true;
    }
    void load(int idx) { full[R::bar(idx)].arrive(1, "a load", idx); landing.push_back(idx); some(); }
    void load_k(int idx, int) { load(idx); }
    void load_v(int idx, int) { load(idx); }
    void pre_k(int idx, int) { load(idx); }
    bool load_q() { return !abort_now; }
};

template <int NS, bool PRE>
void walk(const std::vector<Item>& items, unsigned seed, bool late, int abort_at) {
    World<NS> w(items, seed, late, abort_at);
    int idx = 0;
    rowmax::kv_begin(w);
    bool ok = true;
    for (const Item& it : items)
        if (ok) ok = rowmax::kv_item<PRE>(w, idx, it.pre, it.n);
    rowmax::kv_end(w, idx);
    if (ok) {
        while (w.consume() || w.land()) {}
        if (w.at != w.mma.size() || !w.landing.empty()) throw Failure{"the MMA warp does not get to the end"};
    } else {
        // The waits at the end: every copy under way belongs to a position that is waited for, and landing ends the phase.
        for (int l : w.landing) {
            bool covered = false;
            for (int i = rowmax::kv_drain_from<NS>(idx); i < idx; ++i) covered = covered || ((i + 1) >> 1) == ((l + 1) >> 1);
            if (!covered) throw Failure{"a copy under way at position " + std::to_string(l) + " is not waited for at the end"};
        }
        while (w.land()) {}
        for (int i = rowmax::kv_drain_from<NS>(idx); i < idx; ++i)
            if (!w.full[KvRing<NS>::bar(i)].done(KvRing<NS>::ph_full(i))) throw Failure{"the wait at the end for position " + std::to_string(i) + " runs out"};
    }
}

template <int NS, bool PRE>
void all(const std::vector<Item>& items, int seeds) {
    int steps = 0;
    for (const Item& it : items) steps += it.pre + 2 * it.n;
    for (int abort_at = -1; abort_at < steps; ++abort_at)
        for (int s = 0; s <= seeds; ++s) {
            try {
                walk<NS, PRE>(items, s, s == 0, abort_at);
            } catch (const Failure& f) {
                std::string list;
                for (const Item& it : items) list += " " + std::to_string(it.pre) + "+" + std::to_string(it.n);
                std::printf("%d slots, items (maxima pass + tiles)%s, gives up at wait %d, seed %d: %s\n", NS, list.c_str(), abort_at, s, f.what.c_str());
                std::exit(1);
            }
        }
}

}  // namespace

int main(int argc, char** argv) {
    const int seeds = argc > 1 ? std::atoi(argv[1]) : 20;
    for (int n = 0; n <= 20; ++n) {
        for (int pre = 0; pre <= 20; ++pre) {       // split form: one item
            all<4, true>({{pre, n}}, seeds);
            all<8, true>({{pre, n}}, seeds);
        }
        for (int second = 0; second <= 6; ++second) {
            all<4, false>({{0, n}, {0, second}, {0, 3}}, seeds);
            all<8, false>({{0, n}, {0, second}, {0, 3}}, seeds);
        }
    }
    std::puts("ok");
    return 0;
}
