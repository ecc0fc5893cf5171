// The ring of K/V tiles between the TMA producer and the MMA warp of attn_fwd_kernel.cuh: which barrier a position has, and the
// producer's order of waits, loads and arrivals.  No CUDA in here but the qualifiers, so that tests/kv_ring_model.cpp can walk
// the same code on the CPU against a model of the barriers.
#pragma once

#ifdef __CUDACC__
#define ROWMAX_HD __host__ __device__ __forceinline__
#else
#define ROWMAX_HD inline
#endif

namespace rowmax {

// Ring positions count tiles over all items: K(0), V(0), K(1), V(1), ...  V(j) and K(j + 1), positions 2i - 1 and 2i, are pair i
// and share a full and an empty barrier: the MMA warp needs both at once and is done with both at once.  (The last V of an item
// goes with the first K of the next.)  A full barrier takes two arrivals a phase, one for each position of its pair.
template <int NS>
struct KvRing {
    static constexpr int kPairs = NS / 2;
    static ROWMAX_HD constexpr int bar(int idx) { return ((idx + 1) >> 1) % kPairs; }
    static ROWMAX_HD constexpr int ph_full(int idx) { return (((idx + 1) >> 1) / kPairs) & 1; }
    static ROWMAX_HD constexpr int ph_empty(int idx) { return ph_full(idx) ^ 1; }
};

// The producer's walk.  Ops:
//   void arrive(idx)                  one arrival on the full barrier of position idx
//   bool wait_empty(idx)              waits for the empty barrier of idx; false: give up, nothing more is to be loaded
//   void load_k(idx, j), load_v(idx, j), pre_k(idx, j)   arrival with the bytes of a tile, and its copies
//   bool load_q()                     the item's query tiles
// Every arrival on a full barrier but the first follows wait_empty for that position: it tells that the pair which had the
// barrier before has landed and been read.  An arrival without it could fall into that pair's phase, whose two arrivals are
// made when its copies are issued: one too many, which an mbarrier does not define.
template <class Ops>
ROWMAX_HD void kv_begin(Ops& ops) { ops.arrive(0); }      // pair 0 has no V

// One item: pre_max tiles of K alone (the maxima pass of the split form), then n_max tiles of K and V.  False: gave up.
template <bool PRE, class Ops>
ROWMAX_HD bool kv_item(Ops& ops, int& idx, int pre_max, int n_max) {
    if constexpr (PRE) {
        for (int j = 0; j < pre_max; ++j) {
            if (!ops.wait_empty(idx)) return false;
            ops.pre_k(idx, j);
            ++idx;
            if (j == 0 && !ops.load_q()) return false;
        }
        if (idx & 1) {     // an odd number of tiles: the position that V would have stays empty
            if (!ops.wait_empty(idx)) return false;
            ops.arrive(idx);
            ++idx;
        }
    }
    // K first: the last P V of the item before waits for it along with its V; then Q, once its buffers are free
    for (int j = 0; j < n_max; ++j) {
        if (!ops.wait_empty(idx)) return false;
        ops.load_k(idx, j);
        ++idx;
        if ((!PRE || pre_max == 0) && j == 0 && !ops.load_q()) return false;
        if (!ops.wait_empty(idx)) return false;
        ops.load_v(idx, j);
        ++idx;
    }
    return true;
}

// After the last item: the last pair is complete without a K.  At an odd position the producer gave up between K and V: the
// pair of that position has not been waited for and nothing is loaded into it.
template <class Ops>
ROWMAX_HD void kv_end(Ops& ops, int idx) {
    if ((idx & 1) == 0) ops.arrive(idx);
}

// First position of those that may still have copies under way when the producer ends at idx.
template <int NS>
ROWMAX_HD constexpr int kv_drain_from(int idx) { return idx >= NS ? idx - NS + 1 : 0; }

// ---- The ring of the two-stream form (attn_streams_kernel.cuh).  Tiles G = 0, 1, ... are counted over all items.  The MMA warp
// needs V(G - 2) and K(G) at once and is done with both at once: they are pair G, whose two slots share a full and an empty
// barrier.  The first two pairs have no V, the two after the last tile no K.
template <int NP>
struct StreamRing {
    static ROWMAX_HD constexpr int bar(int pair) { return pair % NP; }
    static ROWMAX_HD constexpr int ph_full(int pair) { return (pair / NP) & 1; }
    static ROWMAX_HD constexpr int ph_empty(int pair) { return ph_full(pair) ^ 1; }
    static ROWMAX_HD constexpr int slot_v(int pair) { return 2 * (pair % NP); }
    static ROWMAX_HD constexpr int slot_k(int pair) { return 2 * (pair % NP) + 1; }
};
// Ops: arrive(pair), wait_empty(pair), load_k(pair), load_v(pair), with the meaning they have above.  False: the producer gave up.
template <class Ops>
ROWMAX_HD bool stream_tile(Ops& ops, int pair) {
    if (!ops.wait_empty(pair)) return false;
    if (pair >= 2) ops.load_v(pair);
    else ops.arrive(pair);
    ops.load_k(pair);
    return true;
}
template <class Ops>
ROWMAX_HD bool stream_tail(Ops& ops, int pair) {
    if (pair < 2) return true;
    if (!ops.wait_empty(pair)) return false;
    ops.load_v(pair);
    ops.arrive(pair);
    return true;
}
// Whether anything arrives for a pair up to the second one after the last of `tiles` tiles.
ROWMAX_HD constexpr bool stream_pair_is_used(int pair, int tiles) { return pair < tiles || pair >= 2; }

template <class Arrive, class WaitEmpty, class LoadK, class LoadV>
struct StreamOps {
    Arrive arrive;
    WaitEmpty wait_empty;
    LoadK load_k;
    LoadV load_v;
};
template <class A, class W, class K, class V>
StreamOps(A, W, K, V) -> StreamOps<A, W, K, V>;

// Ops out of callables.
template <class Arrive, class WaitEmpty, class LoadK, class LoadV, class PreK, class LoadQ>
struct KvOps {
    Arrive arrive;
    WaitEmpty wait_empty;
    LoadK load_k;
    LoadV load_v;
    PreK pre_k;
    LoadQ load_q;
};
template <class A, class W, class K, class V, class P, class Q>
KvOps(A, W, K, V, P, Q) -> KvOps<A, W, K, V, P, Q>;

}  // namespace rowmax
