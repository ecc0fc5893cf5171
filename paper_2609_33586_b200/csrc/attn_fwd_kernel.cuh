// Fused attention forward for sm_100a: TMA-staged Q/K/V tiles, tcgen05 MMAs with TMEM accumulators,
// online softmax with a selectable weight map (exact / Rowmax-PoT / Rowmax-H15), bf16 O + fp32 LSE.
//
// Loop structure per query tile (Sec. 5.2; App. B.1): for each key tile in ascending order
//   S = Q K^T -> tile row maximum -> running maximum m (always adopted, threshold 0) ->
//   x = s*c - m*c -> weight map -> row sum l and P (same weights) -> O = alpha*O + P V;
// at the end O = v_descale * O / l and LSE = ln2 * (m*c + log2 l).
//
// Persistent grid: one CTA (16 warps) per SM walks work items, each a pair of query tiles of 128 rows
// of one (batch, head) whose key tiles it visits once, so every K/V tile staged in shared memory
// feeds four MMAs:
//   warpgroup 0/1  softmax of query tile 0/1: one thread per row (no shuffles needed: a thread
//                  reads its whole score row from TMEM), weight map, row sum, P written back to
//                  TMEM over the S columns; after the last key tile the epilogue of its rows
//   warpgroup 2    correction: rescales the O accumulators in TMEM when a running maximum moved
//   warp 12        MMA issuer (one thread): S_t = Q_t K^T and O_t += P_t V on the tensor cores
//   warp 13        TMA producer (one thread): Q per item, K/V through a ring of shared-memory slots
// While warpgroup 0 works on S_0(j), the tensor cores compute P_1 V(j-1) and S_1(j), and vice versa.
//
// What bounds it: at 16 bits the MMA warp.  Issuing blocks until the tensor cores take the instruction (eight bf16 MMAs of
// 128 x 128 x 16: 520 clocks), and every barrier it waits for costs 100 to 150 clocks even when it is ready, in which the tensor
// cores idle; so P and the rescaled O share a barrier, V(j) and K(j + 1) share theirs, and O is committed once per item
// (bf16 8K h15 267 -> 247 us).  At fp8 the chain of one softmax warpgroup (about 1500 clocks of work, 1000 until its next
// scores are there).
// Split form (SPLIT): when there are fewer items than SMs a cluster of CTAs shares an item, each taking a contiguous part
// of its key tiles.  Every part must start with the anchor the sequential loop would have reached there, so for the rounding
// maps the cluster first goes over all parts but the last for the row maxima alone (Q K^T and a maximum, two thirds of a
// full step).  Exact-like modes on 16-bit inputs need no such pass; on fp8 inputs the rounding of P to e4m3 depends on the
// anchor, and the result should not depend on the split.  At the end each CTA leaves
// O, l and its anchor in shared memory and adds up its share of the rows over the cluster.
// TMEM columns: S_0/P_0 [0,128), S_1/P_1 [128,256), O_0 [256,384), O_1 [384,512).
#pragma once
#include "kv_ring.cuh"
#include "plan.h"
#include "softmax_math.cuh"

namespace rowmax {

namespace {

// Whether the parts of a split item need the row maxima of the parts before them.
__host__ __device__ constexpr bool split_takes_maxima(int mode, bool fp8) { return fp8 || !is_exact_like(mode); }

template <int D, bool FP8, bool SPLIT = false>
struct WsCfg {
    using C = TileCfg<D, FP8>;
    static constexpr int kSlots = FP8 ? 8 : (D == 128 ? 4 : 8);  // K/V ring slots (one tile each)
    static constexpr int kQBytes = 2 * C::kTileBytes;
    static constexpr int kRingBytes = kSlots * C::kTileBytes;
    static constexpr int kScaleOff = kQBytes + kRingBytes;        // float alpha[2][128]
    static constexpr int kBarOff = kScaleOff + 2 * 128 * 4;
    static constexpr int kNumBars = 2 * kSlots + 7 * 2 + 1 + (SPLIT ? 2 + 2 + 3 : 0);
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    // split form: row maxima of the parts before this one, [part][256]; anchor and row sum of this part, [256][2]; weights of
    // the parts for the rows this CTA adds up, [part][rows]
    static constexpr int kXmaxOff = kMiscOff + 16;
    static constexpr int kMlOff = kXmaxOff + (SPLIT ? (kMaxSplit - 1) * 256 * 4 : 0);
    static constexpr int kPartWOff = kMlOff + (SPLIT ? 256 * 8 : 0);
    static constexpr int kEndOff = kPartWOff + (SPLIT ? (256 + kMaxSplit) * 4 : 0);
    static constexpr int kSmemBytes = kEndOff + 1024;             // + manual 1024-byte alignment slack
    static_assert(!SPLIT || 2 * kTileM * D * 4 <= kQBytes + kRingBytes, "O of both tiles is parked over Q and the ring");
    static_assert(kSmemBytes <= 232448, "exceeds the 227 KB shared memory of an sm_100 CTA");
};

// Register split of the 512 threads x 128 registers the CTA is launched with (setmaxnreg can only
// redistribute that allocation; a larger total would make the increase wait for ever): softmax /
// correction / MMA+TMA warpgroups.  The softmax warps hold a row of 128 scores; what decides is that no role spills: with
// 192 / 80 / 48 and a correction that took 32 columns at a time the 16-bit instances spilled in the MMA and correction
// warps and were 2 to 4 % slower (bf16 8K exact, full-attention fp8 exact; both in turn on one machine, SM clock not recorded);
// 208 / 48 / 48 spills again (7 % slower).
constexpr int kRegSoftmax = 200, kRegCorr = 56, kRegMma = 56;
static_assert(256 * kRegSoftmax + 128 * kRegCorr + 128 * kRegMma <= 512 * 128, "setmaxnreg targets exceed the launch allocation");
template <int N> __device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

// Optional cycle stamps (compiled in only with -DROWMAX_TRACE): one representative thread per role of
// one chosen CTA writes clock64() at fixed points of its first 64 key tiles.
#ifdef ROWMAX_TRACE
#define ROWMAX_STAMP(role, j, slot)                                                              \
    do {                                                                                         \
        if (p.trace != nullptr && static_cast<int>(blockIdx.x) == p.trace_block && (j) < 64)     \
            p.trace[((role) * 64 + (j)) * 8 + (slot)] = clock64();                               \
    } while (0)
#else
#define ROWMAX_STAMP(role, j, slot) do { } while (0)
#endif

constexpr int kBarSelftest = 0x7F;
constexpr int kBarAlign = 0x7E;      // not a barrier: the shared memory of the launch is not aligned as declared
enum BarId : int { kBarQFull = 0, kBarQEmpty = 1, kBarKvFull = 2, kBarKvEmpty = 3, kBarSFull = 4, kBarPFull = 5,
                   kBarOFull = 6, kBarScale = 7, kBarFin = 8, kBarOFree = 9,
                   kBarSFree = 10, kBarXmax = 11, kBarPart = 12, kBarItem = 13 };

// One work item = two query tiles of 128 rows of one (batch, head).
struct WorkItem {
    int h, b, hk;
    int q0[2];   // first query row of each tile
    int n[2];    // key tiles of each tile (0: the tile is out of range or sees no key), split form: of this CTA's part
    int n_max;
    int j0;      // first key tile (0 but in the split form)
    // split form, maxima pass: first key tile, key tiles of each query tile
    int pre_j0, pre_n[2];
};

// Items are numbered heaviest first (under a causal mask the last query tiles have the most key
// tiles).  CTA c of G walks them in a snake: round k takes item k*G + c (k even) or k*G + G-1-c (k odd),
// so every CTA gets one item of each weight class and the loads even out without a global counter.
__device__ __forceinline__ int item_index(int round, int cta, int n_ctas) {
    return round * n_ctas + ((round & 1) ? (n_ctas - 1 - cta) : cta);
}
__device__ __forceinline__ WorkItem decode_item(int w, const AttnParams& p, int n_pairs, int bh) {
    WorkItem it;
    const int pair = n_pairs - 1 - w / bh;
    const int rem = w % bh;
    it.h = rem % p.Hq;
    it.b = rem / p.Hq;
    it.hk = it.h / p.group;
    const int shift = p.Sk - p.Sq;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        it.q0[t] = pair * 2 * kTileM + t * kTileM;
        const int kv_end = p.causal ? min(p.Sk, it.q0[t] + kTileM + shift) : p.Sk;
        it.n[t] = (it.q0[t] < p.Sq && kv_end > 0) ? (kv_end + kTileN - 1) / kTileN : 0;
    }
    it.n_max = max(it.n[0], it.n[1]);
    it.j0 = it.pre_j0 = it.pre_n[0] = it.pre_n[1] = 0;
    return it;
}
// Part `rank` of `parts` of an item: key tiles [j0, j0 + n[t]) of each query tile, and of the maxima pass key tiles
// [pre_j0, pre_j0 + pre_n[t]): the CTA's own part unless it is the last, whose maxima nobody needs; with two parts each CTA
// takes half of the first one.
__device__ __forceinline__ WorkItem part_of_item(WorkItem it, int rank, int parts) {
    const int full[2] = {it.n[0], it.n[1]};
    const int j1 = (rank + 1) * it.n_max / parts;
    it.j0 = rank * it.n_max / parts;
    const int half = it.n_max / 2;
    it.pre_j0 = parts == 2 ? (rank == 0 ? 0 : half / 2) : it.j0;
    const int pre_j1 = parts == 2 ? (rank == 0 ? half / 2 : half) : (rank == parts - 1 ? it.j0 : j1);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        it.n[t] = max(0, min(full[t], j1) - it.j0);
        it.pre_n[t] = max(0, min(full[t], pre_j1) - it.pre_j0);
    }
    it.n_max = max(it.n[0], it.n[1]);
    return it;
}

}  // namespace

// IN: storage type of q, k, v (kInBF16 / kInFP8 / kInFP16).  P has the type of V at 16 bits (the f16
// kind wants both MMA operands in one format) and one of the two fp8 formats at 8 bits.
// TAU: deferred rescale (attn_fwd_tau, bf16 only), an instance of its own: the adoption rule in the common instances cost
// them 1.5 to 3.5 % (bf16 8K h15 251.0 -> 244.3 us without).
template <int D, int IN, int MODE, bool SPLIT = false, bool TAU = false>
__global__ void __launch_bounds__(512, 1)
attn_fwd_ws_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr bool FP8 = IN == kInFP8;
    constexpr bool HALF = IN == kInFP16;
    using C = TileCfg<D, FP8>;
    using W = WsCfg<D, FP8, SPLIT>;
    constexpr int NS = W::kSlots;
    constexpr bool kOutOfStep = FP8 && is_exact_like(MODE);   // keep the softmax warpgroups apart (see below)
    constexpr bool kPre = SPLIT && split_takes_maxima(MODE, FP8);   // row maxima of the part first
    // Declared with the alignment that the swizzled tiles need: all shared-memory addresses are then constants, not
    // registers, of which the softmax warps have none to spare (checked below).
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sQ = smem_u32(smem);
    const uint32_t sRing = sQ + W::kQBytes;
    const uint32_t sScale = smem_u32(smem + W::kScaleOff);
    const uint32_t bar0 = smem_u32(smem + W::kBarOff);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + W::kMiscOff);
    const uint32_t abort_at = smem_u32(smem + W::kMiscOff + 4), leave_at = smem_u32(smem + W::kMiscOff + 8);
    const WaitCtx wctx{abort_at, p.status, kWaitLimitCycles};

    // barrier addresses
    // ring positions, pairs of them and the order of waits and arrivals: kv_ring.cuh
    using Ring = KvRing<NS>;
    constexpr int NP = Ring::kPairs;
    auto bar_kv_full = [&](int idx) { return bar0 + 8u * Ring::bar(idx); };
    auto bar_kv_empty = [&](int idx) { return bar0 + 8u * (NS + Ring::bar(idx)); };
    auto ph_kv_full = [&](int idx) { return Ring::ph_full(idx); };
    auto ph_kv_empty = [&](int idx) { return Ring::ph_empty(idx); };
    auto bar_x = [&](int which, int t) { return bar0 + 8u * (2 * NS + 2 * which + t); };
    auto bar_q_full = [&](int t) { return bar_x(0, t); };      // TMA -> MMA: Q_t of the current item landed
    auto bar_q_empty = [&](int t) { return bar_x(1, t); };     // MMA -> TMA: last S_t MMA of the item done
    auto bar_s_full = [&](int t) { return bar_x(2, t); };      // MMA -> softmax: S_t(j) is in TMEM
    auto bar_p_full = [&](int t) { return bar_x(3, t); };      // softmax and correction -> MMA: P_t(j) is in TMEM, O_t rescaled
    auto bar_o_full = [&](int t) { return bar_x(4, t); };      // MMA -> epilogue: the last P_t V of the item accumulated
    auto bar_scale = [&](int t) { return bar_x(5, t); };       // softmax -> correction: alpha_t(j) in smem
    auto bar_o_free = [&](int t) { return bar_x(6, t); };      // epilogue -> MMA: O_t has been read out
    const uint32_t bar_drain = bar0 + 8u * (2 * NS + 14);      // abort path only: the MMA warp's last commit
    // split form.  The maxima pass has two score buffers per query tile: S_t and, as O_t is not in use yet, O_t; the two tiles
    // go through it together (one wait and one commit for both; 512 queries on 16K, bf16 h15: 147 -> 142 us).
    auto bar_pre_free = [&](int b) { return bar0 + 8u * (2 * NS + 15 + b); };   // softmax -> MMA: buffer b of both tiles has been read
    auto bar_pre_full = [&](int b) { return bar0 + 8u * (2 * NS + 17 + b); };   // MMA -> softmax: scores of both tiles in buffer b
    const uint32_t bar_xmax = bar0 + 8u * (2 * NS + 19);       // the maxima of all parts before this one are here
    const uint32_t bar_item = bar0 + 8u * (2 * NS + 20);       // MMA -> softmax: all products of the item are complete
    const uint32_t bar_part = bar0 + 8u * (2 * NS + 21);       // all parts have left O, l and anchor

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wg = warp >> 2;
    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicCAS(p.status, 0, (kRoleSetup << 8) | kBarAlign);
        return;
    }
    // The status word is sticky: once a wait has expired (in an earlier launch, or in another CTA of this one) and
    // until the host clears it, a CTA that starts is a no-op: it touches neither its outputs nor TMEM nor TMA.
    // One thread reads the word, and what it read is kept in a place of its own (leave_at), so that the whole CTA takes the
    // same way: abort_at may be set by a role while slower warps are still on their way to theirs.
    if (tid == 0) {
        const int set = *reinterpret_cast<volatile int*>(p.status) != 0 ? 1 : 0;
        write_flag(abort_at, set);
        write_flag(leave_at, set);
    }
#ifdef ROWMAX_TRACE
    const long long trace_t0 = clock64();
#endif
    if (tid == 256) ROWMAX_STAMP(2, 63, 0);

    const int n_pairs = (p.Sq + 2 * kTileM - 1) / (2 * kTileM);
    const int bh = p.Hq * p.B;
    const int n_items = n_pairs * bh;
    const int parts = SPLIT ? p.split : 1, rank = SPLIT ? static_cast<int>(cluster_ctarank()) : 0;
    const int cta = SPLIT ? blockIdx.x / parts : blockIdx.x, n_ctas = SPLIT ? gridDim.x / parts : gridDim.x;
    const int shift = p.Sk - p.Sq;

    if (warp == 13) {
        if (lane < NP) {
            mbar_init(bar0 + 8u * lane, 2);            // V(j) and K(j + 1)
            mbar_init(bar0 + 8u * (NS + lane), 1);
        } else if (lane >= 16 && lane < 18) {
            const int t = lane - 16;
            mbar_init(bar_q_full(t), 1);
            mbar_init(bar_q_empty(t), 1);
            mbar_init(bar_s_full(t), 1);
            mbar_init(bar_p_full(t), 8);      // one arrival per softmax warp, one per correction warp
            mbar_init(bar_o_full(t), 1);
            mbar_init(bar_scale(t), 4);
            mbar_init(bar_o_free(t), 4);      // one arrival per softmax warp (epilogue)
        } else if (lane == 18) {
            mbar_init(bar_drain, 1);
        } else if (SPLIT && lane == 19) {
            for (int i = 0; i < 2; ++i) {
                mbar_init(bar_pre_free(i), 8);      // one arrival per softmax warp of both tiles
                mbar_init(bar_pre_full(i), 1);
            }
            mbar_init(bar_item, 1);
            mbar_init(bar_xmax, rank > 0 ? 8 * rank : 1);   // one per softmax warp of each part before
            mbar_init(bar_part, 8 * parts);   // one per softmax warp of every part
        }
        fence_mbar_init();
    }
    constexpr uint32_t kTmemCols = 512;
    if (warp == 12) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // Everything above is the CTA's own; what follows reads the caller's tensors, which the kernel before this one in the
    // stream may still be writing.
    griddep_wait();
    griddep_launch();
    if constexpr (SPLIT) {
        // The others of the cluster reach into this CTA's shared memory: every CTA takes all steps, with waits that end soon
        // if the flag is set, and leaves with the cluster.
        cluster_arrive();
        cluster_wait();
    } else if (flag_is_set(leave_at)) {
        if (warp == 12) tmem_dealloc(tmem, kTmemCols);
        return;
    }
    auto get_item = [&](int w) {
        WorkItem it = decode_item(w, p, n_pairs, bh);
        if constexpr (SPLIT) it = part_of_item(it, rank, parts);
        return it;
    };
    if (tid == 256) ROWMAX_STAMP(2, 63, 1);
    auto tmem_S = [&](int t) { return tmem + 128u * t; };
    auto tmem_O = [&](int t) { return tmem + 256u + 128u * t; };

    constexpr uint32_t fmt_16 = HALF ? kFmtF16 : kFmtBF16;
    constexpr uint32_t fmt_ab = FP8 ? kFmtE4M3 : fmt_16;
    constexpr uint32_t fmt_p = FP8 ? (PFormat<FP8, MODE>::kE4M3 ? kFmtE4M3 : kFmtE5M2) : fmt_16;
    constexpr uint32_t idesc_s = umma_idesc(fmt_ab, fmt_ab, false, false, kTileM, kTileN);
    constexpr uint32_t idesc_pv = umma_idesc(fmt_p, fmt_ab, false, true, kTileM, D);
    constexpr float p_off = static_cast<float>(PFormat<FP8, MODE>::kOffLog2);  // log2 of the P / row-sum scale

    if (wg == 3) {
        reg_dec<kRegMma>();
        if (warp == 13 && lane == 0) {
            // ------------------------------------------------------------ TMA producer
            int kv_idx = 0;             // ring position: K/V tiles loaded so far, over all items
            int q_use[2] = {0, 0};      // items that used Q buffer t so far
            WorkItem it;
            auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, uint32_t bar, int head, int row0) {
                mbar_arrive_expect_tx(bar, C::kTileBytes);
#pragma unroll
                for (int bx = 0; bx < C::kBoxes; ++bx)
                    tma_load_4d(dst + bx * C::kBoxBytes, tm, bar, bx * C::kBoxElems, head, row0, it.b);
            };
            auto load_kv = [&](const CUtensorMap* tm, int idx, int tile) {
                load_tile(tm, sRing + (idx % NS) * C::kTileBytes, bar_kv_full(idx), it.hk, tile * kTileN);
            };
            // After an expired wait nothing more is loaded: a wait then returns at once, and a copy into a buffer
            // whose last copy may still be under way would leave more in flight than the waits below account for.
            auto load_q = [&](int t) {
                if (it.n[t] > 0 || (kPre && it.pre_n[t] > 0)) {
                    mbar_wait(bar_q_empty(t), (q_use[t] & 1) ^ 1, wctx, (kRoleLoad << 8) | kBarQEmpty);
                    if (flag_is_set(abort_at)) return false;
                    load_tile(&tmQ, sQ + t * C::kTileBytes, bar_q_full(t), it.h, it.q0[t]);
                    ++q_use[t];
                }
                return true;
            };
            KvOps ops{[&](int idx) { mbar_arrive(bar_kv_full(idx)); },
                      [&](int idx) {
                          if constexpr (SPLIT) mbar_wait_poll(bar_kv_empty(idx), ph_kv_empty(idx), wctx, (kRoleLoad << 8) | kBarKvEmpty);
                          else mbar_wait(bar_kv_empty(idx), ph_kv_empty(idx), wctx, (kRoleLoad << 8) | kBarKvEmpty);
                          return !flag_is_set(abort_at);
                      },
                      [&](int idx, int j) { load_kv(&tmK, idx, it.j0 + j); },
                      [&](int idx, int j) { load_kv(&tmV, idx, it.j0 + j); },
                      [&](int idx, int j) { load_kv(&tmK, idx, it.pre_j0 + j); },
                      [&]() { return load_q(0) && load_q(1); }};
            kv_begin(ops);
            for (int round = 0; !SPLIT || round < 1; ++round) {   // split form: one item per cluster
                const int w = item_index(round, cta, n_ctas);
                if (w >= n_items) break;
                it = get_item(w);
                if (round == 0) ROWMAX_STAMP(3, 63, 0);
                if (!kv_item<kPre>(ops, kv_idx, kPre ? max(it.pre_n[0], it.pre_n[1]) : 0, it.n_max)) break;
            }
            kv_end(ops, kv_idx);
            // Before the CTA ends every load this thread issued must have landed.  Normally the consumers have
            // seen to that and these waits return at once; after an expired wait they may have stopped waiting while
            // copies were still writing shared memory, so wait (bounded) for the last use of every pair of ring slots and
            // Q buffer.
            for (int idx = kv_drain_from<NS>(kv_idx); idx < kv_idx; ++idx)
                mbar_wait_quiet(bar_kv_full(idx), ph_kv_full(idx), kDrainLimitCycles);
#pragma unroll
            for (int t = 0; t < 2; ++t)
                if (q_use[t] > 0) mbar_wait_quiet(bar_q_full(t), (q_use[t] - 1) & 1, kDrainLimitCycles);
        } else if (warp == 12) {
            // ------------------------------------------------------------ MMA issuer
            // The whole warp walks the loop (so addresses and descriptors stay warp-uniform values);
            // one elected lane issues the MMAs and commits.
            const bool leader = elect_one();
            constexpr uint32_t desc_hi = umma_desc_hi_sw(C::kSwizzle);
            const uint32_t q_lo0 = umma_desc_lo(sQ, 16);
            const uint32_t ring_lo_k = umma_desc_lo(sRing, 16);               // K tiles: K-major
            const uint32_t ring_lo_v = umma_desc_lo(sRing, C::kBoxBytes);     // V tiles: MN-major, LBO = next 128-byte column block
            constexpr uint32_t kTileLo = C::kTileBytes >> 4;
            auto issue_s = [&](int t, uint32_t k_lo, uint32_t dst) {
                const uint32_t q_lo = q_lo0 + t * kTileLo;
#pragma unroll
                for (int ks = 0; ks < C::kQkSteps; ++ks) {
                    const uint32_t off = ((ks / C::kStepsPerBox) * C::kBoxBytes + (ks % C::kStepsPerBox) * 32) >> 4;
                    umma_ss_lo<FP8>(dst, q_lo + off, k_lo + off, desc_hi, idesc_s, ks > 0 ? 1u : 0u);
                }
            };
            auto issue_pv = [&](int t, uint32_t v_lo, bool accumulate) {
#pragma unroll
                for (int ks = 0; ks < C::kPvSteps; ++ks) {
                    const uint32_t off = (ks * C::kUmmaK * C::kSwizzle) >> 4;   // kUmmaK keys down the MN-major V tile
                    umma_ts_lo<FP8>(tmem_O(t), tmem_S(t) + ks * 8, v_lo + off, desc_hi, idesc_pv,
                                    (accumulate || ks > 0) ? 1u : 0u);
                }
            };
            auto slot_lo = [&](int idx) { return static_cast<uint32_t>(idx % NS) * kTileLo; };
            auto wait_full = [&](int idx) {
                mbar_wait(bar_kv_full(idx), ph_kv_full(idx), wctx, (kRoleMma << 8) | kBarKvFull);
            };
            int kv_base = 0;            // ring index of K_0 of the current item
            int tiles[2] = {0, 0};      // key tiles of query tile t finished in earlier items (barrier phases)
            int q_use[2] = {0, 0};      // items that used Q buffer / O accumulator t so far
            for (int round = 0; !SPLIT || round < 1; ++round) {   // split form: one item per cluster
                const int w = item_index(round, cta, n_ctas);
                if (w >= n_items) break;
                const WorkItem it = get_item(w);
                if constexpr (kPre) {
                    const int pre_max = max(it.pre_n[0], it.pre_n[1]);
                    for (int j = 0; j < pre_max; ++j) {
                        if (kv_base == 0 || (kv_base & 1)) mbar_wait_poll(bar_kv_full(kv_base), ph_kv_full(kv_base), wctx, (kRoleMma << 8) | kBarKvFull);
                        const int buf = j & 1;
                        if (j == 0) {
#pragma unroll
                            for (int t = 0; t < 2; ++t)
                                if (it.pre_n[t] > 0) mbar_wait(bar_q_full(t), q_use[t] & 1, wctx, (kRoleMma << 8) | kBarQFull);
                        }
                        if (j >= 2) mbar_wait_poll(bar_pre_free(buf), (j / 2 - 1) & 1, wctx, (kRoleMma << 8) | kBarSFree);
                        tc_fence_after();
                        if (leader) {
                            if (!flag_is_set(abort_at)) {
#pragma unroll
                                for (int t = 0; t < 2; ++t)
                                    if (j < it.pre_n[t]) issue_s(t, ring_lo_k + slot_lo(kv_base), buf == 0 ? tmem_S(t) : tmem_O(t));
                            }
                            umma_commit(bar_pre_full(buf));
                        }
                        if (leader && (kv_base & 1) == 0) umma_commit(bar_kv_empty(kv_base));
                        __syncwarp();
                        ++kv_base;
                    }
                    kv_base += kv_base & 1;
                    if (pre_max > 0) {     // both buffers have been read: their last uses
                        const int last = pre_max - 1;
                        mbar_wait_poll(bar_pre_free(last & 1), (last / 2) & 1, wctx, (kRoleMma << 8) | kBarSFree);
                        if (last > 0) mbar_wait_poll(bar_pre_free((last - 1) & 1), ((last - 1) / 2) & 1, wctx, (kRoleMma << 8) | kBarSFree);
                    }
                }
                if (it.n_max > 0) {
                    wait_full(kv_base);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        if (it.n[t] > 0) {
                            if (!kPre || it.pre_n[t] == 0)
                                mbar_wait(bar_q_full(t), q_use[t] & 1, wctx, (kRoleMma << 8) | kBarQFull);
                            // spread the two tiles' weight phases apart from the start (D = 64: 199 -> 190 us at 8K)
                            if (kOutOfStep && round == 0 && t == 1 && it.n[0] > 0)
                                mbar_wait(bar_p_full(0), 0, wctx, (kRoleMma << 8) | kBarPFull);
                            tc_fence_after();
                            if (leader) {
                                if (round == 0) ROWMAX_STAMP(3, 63, 1 + t);
                                if (!flag_is_set(abort_at)) issue_s(t, ring_lo_k + slot_lo(kv_base), tmem_S(t));
                                umma_commit(bar_s_full(t));
                                if (it.n[t] == 1) umma_commit(bar_q_empty(t));
                            }
                        }
                    }
                    if (leader) umma_commit(bar_kv_empty(kv_base));
                    for (int j = 0; j < it.n_max; ++j) {
                        // Everything the next MMAs need besides P is awaited first (it is normally there long
                        // before), so that once P_t(j) arrives the P V and next-S MMAs go out back to back.  (The flag
                        // is read here, off that path: if one of the waits below expires, this step's MMAs still go
                        // out, on stale operands; nothing is stored after that and the MMAs are awaited at the end.)
                        const bool ok = !flag_is_set(abort_at);
                        wait_full(kv_base + 2 * j + 1);      // V(j) and K(j + 1)
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            if (j < it.n[t]) {
                                const uint32_t ph = (tiles[t] + j) & 1;
                                // the accumulator of the previous item must have been read out
                                if (j == 0) mbar_wait(bar_o_free(t), (q_use[t] & 1) ^ 1, wctx, (kRoleMma << 8) | kBarOFree);
                                mbar_wait_poll(bar_p_full(t), ph, wctx, (kRoleMma << 8) | kBarPFull);
                                if (leader) ROWMAX_STAMP(3, j, t * 4 + 0);
                                tc_fence_after();
                                if (leader) {
                                    if (ok) issue_pv(t, ring_lo_v + slot_lo(kv_base + 2 * j + 1), j > 0);
                                    if (j + 1 == it.n[t]) umma_commit(bar_o_full(t));
                                    ROWMAX_STAMP(3, j, t * 4 + 2);
                                    if (j + 1 < it.n[t]) {
                                        if (ok) issue_s(t, ring_lo_k + slot_lo(kv_base + 2 * j + 2), tmem_S(t));
                                        umma_commit(bar_s_full(t));
                                        if (j + 2 == it.n[t]) umma_commit(bar_q_empty(t));   // last S of this item
                                        ROWMAX_STAMP(3, j, t * 4 + 3);
                                    }
                                }
                            }
                        }
                        // V(j) and K(j + 1); V of the last tile goes with K(0) of the next item
                        if (leader && j + 1 < it.n_max) umma_commit(bar_kv_empty(kv_base + 2 * j + 2));
                        __syncwarp();
                    }
                }
                if constexpr (SPLIT) {
                    if (leader) umma_commit(bar_item);
                    __syncwarp();
                }
                kv_base += 2 * it.n_max;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    tiles[t] += it.n[t];
                    if (it.n[t] > 0) ++q_use[t];
                }
            }
            // No MMA of this thread may still be running when TMEM is handed back: one last commit, awaited with a
            // bound (it arrives at once unless a wait expired and the roles left their loops early).
            if (leader) umma_commit(bar_drain);
            mbar_wait_quiet(bar_drain, 0, kDrainLimitCycles);
        }
    } else if (wg == 2) {
        // ---------------------------------------------------------------- correction
        reg_dec<kRegCorr>();
        const int r = tid & 127;
        const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
        int tiles[2] = {0, 0};
        for (int round = 0; !SPLIT || round < 1; ++round) {   // split form: one item per cluster
            const int w = item_index(round, cta, n_ctas);
            if (w >= n_items) break;
            const WorkItem it = get_item(w);
            for (int j = 0; j < it.n_max; ++j) {
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (j < it.n[t]) {
                        mbar_wait(bar_scale(t), (tiles[t] + j) & 1, wctx, (kRoleCorr << 8) | kBarScale);
                        if (r == 0) ROWMAX_STAMP(2, j, t * 4 + 0);
                        const float alpha = ld_shared_f32(sScale + (t * 128 + r) * 4);
                        if (j > 0) {
                            // P V(j - 1) is complete: the softmax warps post alpha(j) after they have seen S(j), whose commit
                            // covers everything issued before it
                            if (r == 0) ROWMAX_STAMP(2, j, t * 4 + 1);
                            __syncwarp();
                            tc_fence_after();
                            if (__any_sync(0xffffffffu, alpha != 1.0f)) {
#pragma unroll
                                for (int cc = 0; cc < D / 16; ++cc) {
                                    uint32_t o[16];
                                    tmem_ld16(tmem_O(t) + lane_base + cc * 16, o);
                                    tmem_wait_ld();
#pragma unroll
                                    for (int i = 0; i < 16; i += 2) {
                                        const float2 v = fmul2(make_float2(__uint_as_float(o[i]), __uint_as_float(o[i + 1])), make_float2(alpha, alpha));
                                        o[i] = __float_as_uint(v.x);
                                        o[i + 1] = __float_as_uint(v.y);
                                    }
                                    tmem_st16(tmem_O(t) + lane_base + cc * 16, o);
                                }
                                tmem_wait_st();
                            }
                            tc_fence_before();
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_p_full(t));
                        if (r == 0) ROWMAX_STAMP(2, j, t * 4 + 2);
                    }
                }
            }
            tiles[0] += it.n[0];
            tiles[1] += it.n[1];
        }
    } else {
        // ---------------------------------------------------------------- softmax + epilogue of query tile t
        reg_inc<kRegSoftmax>();
        // The kernel before this one may have set the status word after the check above.  Each of the warps that store looks
        // again for itself, while it would wait for its first scores.
        if (lane == 0 && *reinterpret_cast<volatile int*>(p.status) != 0) write_flag(abort_at, 1);
        __syncwarp();
        const int t = wg;
        const int r = tid & 127;
        const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_S(t) + lane_base;
        const uint32_t tO = tmem_O(t) + lane_base;
        constexpr int kFam = h15_family_k(MODE);   // h15 family: the map takes the offset times 2^kFam
        const float c_eff = static_cast<float>(1 << kFam) * p.c;
        // 16-bit inputs: the h15 family uses the saturating form of weights_chunk32 (no row-minimum pass, no
        // clamped or masked variants) whenever the anchor is always current (offsets <= 0); the deferred rescale,
        // where a score may lie above its anchor, keeps the form with explicit clamps.  fp8 inputs keep the
        // packed form: there a bound on the key magnitude already removes the row-minimum pass, and the
        // scalar multiply-adds of the saturating form cost more issue slots than they save (measured 4 to 6 %).
        constexpr bool kLattice = kFam > 0 && !FP8;
        constexpr bool kSatForm = kLattice && !TAU;
        int tiles = 0;
        int o_use = 0;      // items with key tiles so far
        for (int round = 0; !SPLIT || round < 1; ++round) {   // split form: one item per cluster
            const int w = item_index(round, cta, n_ctas);
            if (w >= n_items) break;
            const WorkItem it = get_item(w);
            const int q0 = t == 0 ? it.q0[0] : it.q0[1];
            const int nt = t == 0 ? it.n[0] : it.n[1];
            const int row = q0 + r;
            const int row_limit = p.causal ? min(p.Sk, row + shift + 1) : p.Sk;  // visible keys of this row
            // first key index that some row of this tile cannot see (tile-uniform)
            const int tile_limit = p.causal ? min(p.Sk, q0 + shift + 1) : p.Sk;
            const int j0 = SPLIT ? it.j0 : 0;
            float m_run = -INFINITY, l_run = 0.f;
            if constexpr (kPre) {
                // the row's maxima; those over the parts before this one are the anchor to start from
                const int pre_n = t == 0 ? it.pre_n[0] : it.pre_n[1], pre_max = max(it.pre_n[0], it.pre_n[1]);
                float m_part = -INFINITY;
                for (int j = 0; j < pre_max; ++j) {
                    const int buf = j & 1;
                    mbar_wait_poll(bar_pre_full(buf), (j / 2) & 1, wctx, (kRoleSoftmax << 8) | kBarSFull);
                    __syncwarp();
                    tc_fence_after();
                    uint32_t s[4][32];
                    if (j < pre_n) {
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) tmem_ld32((buf == 0 ? tS : tO) + cc * 32, s[cc]);
                        tmem_wait_ld();
                        tc_fence_before();
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_pre_free(buf));
                    if (j < pre_n) {
                        if ((it.pre_j0 + j + 1) * kTileN > tile_limit) {
                            const int col_limit = row_limit - (it.pre_j0 + j) * kTileN;
#pragma unroll
                            for (int cc = 0; cc < 4; ++cc)
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    if (cc * 32 + i >= col_limit) s[cc][i] = __float_as_uint(-INFINITY);
                        }
                        m_part = fmaxf(m_part, row_max128(s));
                    }
                }
                const uint32_t xmax = smem_u32(smem + W::kXmaxOff) + (t * 128 + r) * 4;
                for (int q = rank + 1; q < parts; ++q) st_cluster_f32(mapa(xmax + rank * 1024, q), m_part);
                __syncwarp();
                if (lane > rank && lane < parts) mbar_arrive_cluster(mapa(bar_xmax, lane));
                if (rank > 0) {
                    if (parts == 2) m_run = m_part;   // of the first part's second half
                    mbar_wait_cluster(bar_xmax, 0, wctx, (kRoleSoftmax << 8) | kBarXmax);
                    __syncwarp();
                    for (int q = 0; q < rank; ++q)
                        m_run = fmaxf(m_run, *reinterpret_cast<const volatile float*>(smem + W::kXmaxOff + q * 1024 + (t * 128 + r) * 4));
                }
            }
            // h15 family at fp8: a lower bound of every raw score of this row that costs nothing per score.
            // |q . k| <= (sum_i |q_i|) * max_i |k_i| and an e4m3 key element is at most 448 in magnitude, so
            // s >= -448 * sum_i |q_i|.  When that bound already keeps the scaled offsets of a tile above the
            // clamp, the tile needs neither the row-minimum pass nor the clamped variant.  The row of Q is
            // read from shared memory (a sum does not care about the swizzle, which stays within the row), which
            // is safe while S_t(1) has not been issued, i.e. for items with at least two key tiles (used from four on).
            float score_floor = -INFINITY;
            if constexpr (FP8 && kFam > 0) {
                if (nt >= 4) {   // the sum costs about three row-minimum passes
                    mbar_wait(bar_s_full(t), tiles & 1, wctx, (kRoleSoftmax << 8) | kBarSFull);   // Q_t has landed
                    score_floor = -448.0f * 1.02f * abs_sum_e4m3_row<D / 16>(sQ + t * C::kTileBytes + r * D);
                }
            }
            for (int j = 0; j < nt; ++j) {
                mbar_wait(bar_s_full(t), (tiles + j) & 1, wctx, (kRoleSoftmax << 8) | kBarSFull);
                if (r == 0) ROWMAX_STAMP(t, j, 0);
                __syncwarp();
                tc_fence_after();
                uint32_t s[4][32];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) tmem_ld32(tS + cc * 32, s[cc]);
                tmem_wait_ld();
                if (r == 0) ROWMAX_STAMP(t, j, 1);

                // Masked scores are set to -inf.  exact: their weight is then 0 by itself.  h15 family: a masked
                // tile takes the clamped variant with the clamp one octave lower, at the input whose
                // weight pattern is +0 (there a real score more than 126 octaves below its anchor also weighs 0,
                // or a denormal, instead of 2^-126: nothing against a row sum >= 1).  pot and the partly emulated
                // exact mode zero the masked weights explicitly (pot's floor 2^-20 is not nothing, and the
                // polynomial route does not take -inf).  Keeping a masked variant out of the common modes
                // makes their hot loop markedly faster.
                const bool masked_tile = (j0 + j + 1) * kTileN > tile_limit;
                const int col_limit = row_limit - (j0 + j) * kTileN;
                if (masked_tile) {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (cc * 32 + i >= col_limit) s[cc][i] = __float_as_uint(-INFINITY);
                }
                const float m_t = row_max128(s);
                // The tile maximum becomes the new anchor when there is none yet or when it exceeds the
                // anchor by more than tau octaves (tau = 0: always, so the anchor is the running maximum).
                float m_new = fmaxf(m_run, m_t);
                if constexpr (TAU) {
                    if (!((m_run == -INFINITY) || ((m_t - m_run) * p.c > p.tau))) m_new = m_run;
                }
                const float m_use = (m_new == -INFINITY) ? 0.f : m_new;
                const float alpha = ex2_approx((m_run - m_use) * p.c);
                m_run = m_new;
                // The rescale factor is posted at once: the correction warps need the whole weight phase.  (Later cost 3 to 8 %.)
                // Only the exact-like modes on fp8 inputs post it after the first 32 weights: posted at once, their two
                // warpgroups fall into step, compete for the special-function unit and then wait together
                // (8K e4m3: causal 437 against 401 us, full attention 454 against 412).
                auto post_alpha = [&]() {
                    st_shared_f32(sScale + (t * 128 + r) * 4, alpha);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_scale(t));
                    if (r == 0) ROWMAX_STAMP(t, j, 2);
                };
                if constexpr (!kOutOfStep) post_alpha();

                // exact: x = s*c - m*c + P offset;  h15 family: scaled input 2^K x = s*(2^K c) - m*(2^K c);  pot: x = s*c - m*c
                RowScale rs;
                float nmc = (is_exact_like(MODE) ? p_off : 0.0f) - m_use * c_eff;
                float c_row = c_eff;
                rs.c = make_float2(c_row, c_row);
                rs.nmc = make_float2(nmc, nmc);
                rs.two22 = p.two22;
                rs.pot_neg_cap = p.pot_neg_cap;
                rs.pot_drop_x = p.pot_drop_x;
                rs.clamp_lo = 0.f;
                if constexpr (kFam > 0) rs.clamp_lo = masked_tile ? h15_clamp_zero<kFam>() : h15_clamp_floor<kFam>();
                float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                if constexpr (kSatForm) {
                    // distance below the anchor as a fraction of the clamp distance R, which is also where a masked
                    // score (-inf) ends up: 2^K * 126 (weight floor 2^-126, Eq. h15), in a tile with masked scores
                    // 2^K * 127 (pattern of +0)
                    constexpr float kR = 126.0f * (1 << kFam), kRm = 127.0f * (1 << kFam);
                    const float big_r = masked_tile ? kRm : kR;
                    const float inv_r = masked_tile ? 1.0f / kRm : 1.0f / kR;
                    rs.su = -c_eff * inv_r;
                    const float ou = (m_use * c_eff) * inv_r;
                    rs.ou = make_float2(ou, ou);
                    rs.sat_mul = -big_r;
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        uint32_t pw[16];
                        weights_chunk32<FP8, MODE, false, true, HALF, true>(s[cc], rs, 32, acc, pw);
                        tmem_st16(tS + cc * 16, pw);
                    }
                } else if (is_pot(MODE) && masked_tile) {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        uint32_t pw[16];
                        weights_chunk32<FP8, MODE, true, true, HALF>(s[cc], rs, col_limit - cc * 32, acc, pw);
                        if constexpr (FP8) tmem_st8(tS + cc * 8, pw);
                        else tmem_st16(tS + cc * 16, pw);
                        if (kOutOfStep && cc == 0) post_alpha();
                    }
                } else {
                    // h15: the clamp is a no-op unless some score of the warp's rows lies more than 126 octaves
                    // below its anchor; the row minimum (one more three-input pass) tells, and the common case
                    // runs without the per-score clamp.  A tile with masked scores always takes the clamp.
                    bool clamp = false;
                    if constexpr (kFam > 0) {
                        if (masked_tile) {
                            clamp = true;
                        } else if (!__all_sync(0xffffffffu, (score_floor - m_use) * c_eff >= -125.0f * (1 << kFam))) {
                            const float lowest = (row_min128(s) - m_use) * c_eff;   // smallest scaled offset of the row
                            clamp = __any_sync(0xffffffffu, !(lowest >= -125.0f * (1 << kFam)));
                        }
                    }
                    if (clamp) {
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            uint32_t pw[16];
                            weights_chunk32<FP8, MODE, false, true, HALF>(s[cc], rs, 32, acc, pw);
                            if constexpr (FP8) tmem_st8(tS + cc * 8, pw);
                            else tmem_st16(tS + cc * 16, pw);
                            if (kOutOfStep && cc == 0) post_alpha();
                        }
                    } else {
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            uint32_t pw[16];
                            weights_chunk32<FP8, MODE, false, false, HALF>(s[cc], rs, 32, acc, pw);
                            if constexpr (FP8) tmem_st8(tS + cc * 8, pw);
                            else tmem_st16(tS + cc * 16, pw);
                            if (kOutOfStep && cc == 0) post_alpha();
                        }
                    }
                }
                const float l_tile = (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
                if (r == 0) ROWMAX_STAMP(t, j, 3);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p_full(t));
                if (r == 0) ROWMAX_STAMP(t, j, 4);
                l_run = l_run * alpha + l_tile;
            }

            if constexpr (SPLIT) {
                // O of this part, unscaled, over Q and the ring: [row of 256][D], 16-byte pieces swizzled by the row.  A part
                // without key tiles leaves no O and says so by its row sum; every other part is added, also where it weighs
                // nothing: as in the loop over all tiles, 0 times an infinity or a NaN shows in O.
                constexpr float kNoPart = -1.0f;
                float2* ml = reinterpret_cast<float2*>(smem + W::kMlOff);
                ml[t * 128 + r] = make_float2(m_run, nt > 0 ? l_run : kNoPart);
                // the products of both query tiles read Q and the ring
                mbar_wait_poll(bar_item, 0, wctx, (kRoleEpi << 8) | kBarItem);
                __syncwarp();
                tc_fence_after();
                constexpr int kPieces = D / 4;
                if (nt > 0) {
                    uint8_t* mine = smem + (t * 128 + r) * (D * 4);
#pragma unroll
                    for (int cc = 0; cc < D / 32; ++cc) {
                        uint32_t o[32];
                        tmem_ld32(tO + cc * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int v4 = 0; v4 < 8; ++v4)
                            *reinterpret_cast<uint4*>(mine + (((cc * 8 + v4) ^ (r & (kPieces - 1))) << 4)) =
                                make_uint4(o[v4 * 4], o[v4 * 4 + 1], o[v4 * 4 + 2], o[v4 * 4 + 3]);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_o_free(t));
                }
                __syncwarp();
                if (lane < parts) mbar_arrive_cluster(mapa(bar_part, lane));
                mbar_wait_cluster(bar_part, 0, wctx, (kRoleEpi << 8) | kBarPart);
                __syncwarp();
                // this CTA's share of the 256 rows, added up over the parts
                const int row_lo = rank * 256 / parts, n_rows = (rank + 1) * 256 / parts - row_lo;
                float* weight = reinterpret_cast<float*>(smem + W::kPartWOff);    // [part][n_rows]
                const int wt = tid;      // 0..255 over both softmax warpgroups
                const float flag = lane < parts ? ld_cluster_f32(mapa(abort_at, lane)) : 0.0f;
                const bool alive = __all_sync(0xffffffffu, __float_as_int(flag) == 0);
                if (wt < n_rows) {
                    const int prow = row_lo + wt, tt = prow >> 7;
                    const int out_row = (tt == 0 ? it.q0[0] : it.q0[1]) + (prow & 127);
                    const uint32_t at = smem_u32(smem + W::kMlOff) + prow * 8;
                    float m_fin = -INFINITY;
                    float2 v[kMaxSplit];
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q) {
                        v[q] = q < parts ? ld_cluster_f32x2(mapa(at, q)) : make_float2(-INFINITY, kNoPart);
                    }
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q) {
                        if (v[q].y > 0.f || v[q].y != v[q].y) m_fin = fmaxf(m_fin, v[q].x);
                    }
                    float l_fin = 0.f;
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q) {
                        // a part without visible keys (no anchor) or with a row sum of zero weighs nothing; a row sum that is no
                        // number makes the row's one
                        const bool weighs = v[q].x != -INFINITY && !(v[q].y <= 0.f);
                        v[q].x = weighs ? ex2_approx((v[q].x - m_fin) * p.c) : 0.f;
                        if (weighs || v[q].y != v[q].y) l_fin += v[q].x * v[q].y;
                    }
                    const bool has_keys = l_fin > 0.f;
                    const float inv = has_keys ? p.v_descale / l_fin : 0.f;
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q)
                        if (q < parts) weight[q * n_rows + wt] = v[q].y == kNoPart ? kNoPart : v[q].x * inv;
                    if (alive && out_row < p.Sq && p.lse != nullptr)
                        p.lse[(static_cast<size_t>(it.b) * p.Hq + it.h) * p.Sq + out_row] =
                            has_keys ? 0.6931471805599453f * (m_fin * p.c + log2f(l_fin) - p_off) : -INFINITY;
                }
                named_barrier<2>(256);
                constexpr int kBatch = 8;      // pieces a thread has in flight from one part
                for (int e0 = wt; e0 < n_rows * kPieces; e0 += 256 * kBatch) {
                    float4 acc[kBatch] = {};
                    for (int q = 0; q < parts; ++q) {
                        float4 v[kBatch];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            const int e = e0 + 256 * u, prow = row_lo + e / kPieces, piece = e % kPieces;
                            if (e < n_rows * kPieces && (prow < 128 ? it.q0[0] : it.q0[1]) + (prow & 127) < p.Sq)
                                v[u] = ld_cluster_f32x4(mapa(smem_u32(smem) + prow * (D * 4) + ((piece ^ (prow & (kPieces - 1))) << 4), q));
                        }
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            const int e = e0 + 256 * u, prow = row_lo + e / kPieces;
                            const bool wanted = e < n_rows * kPieces && (prow < 128 ? it.q0[0] : it.q0[1]) + (prow & 127) < p.Sq;
                            const float wq = wanted ? weight[q * n_rows + e / kPieces] : kNoPart;
                            if (!(wq < 0.f)) {
                                acc[u].x = fmaf(wq, v[u].x, acc[u].x);
                                acc[u].y = fmaf(wq, v[u].y, acc[u].y);
                                acc[u].z = fmaf(wq, v[u].z, acc[u].z);
                                acc[u].w = fmaf(wq, v[u].w, acc[u].w);
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const int e = e0 + 256 * u, prow = row_lo + e / kPieces, piece = e % kPieces;
                        const int out_row = (prow < 128 ? it.q0[0] : it.q0[1]) + (prow & 127);
                        if (alive && e < n_rows * kPieces && out_row < p.Sq) {
                            uint2 pk;
                            pk.x = pack_bf16_rn(acc[u].x, acc[u].y);
                            pk.y = pack_bf16_rn(acc[u].z, acc[u].w);
                            *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.o) +
                                                      ((static_cast<size_t>(it.b) * p.Sq + out_row) * p.Hq + it.h) * D + piece * 4) = pk;
                        }
                    }
                }
            } else
            // epilogue of this tile: O = v_descale * acc / l (the P offset cancels), LSE = ln2 * (m c + log2 l)
            if (q0 < p.Sq) {
                const bool has_keys = (m_run != -INFINITY) && l_run > 0.f;
                const float inv = has_keys ? p.v_descale / l_run : 0.f;
                const bool alive = !flag_is_set(abort_at);      // after an expired wait the accumulators are not to be trusted: store nothing
                if (alive && row < p.Sq && p.lse != nullptr) {
                    const float lse = has_keys ? 0.6931471805599453f * (m_run * p.c + log2f(l_run) - p_off) : -INFINITY;
                    p.lse[(static_cast<size_t>(it.b) * p.Hq + it.h) * p.Sq + row] = lse;
                }
                if (nt > 0) {
                    mbar_wait(bar_o_full(t), o_use & 1, wctx, (kRoleEpi << 8) | kBarOFull);
                    ++o_use;
                    __syncwarp();
                    tc_fence_after();
                }
                if (r == 0 && round == 0) ROWMAX_STAMP(2, 63, 2 + 2 * t);
                __nv_bfloat16* orow = reinterpret_cast<__nv_bfloat16*>(p.o) +
                                      ((static_cast<size_t>(it.b) * p.Sq + row) * p.Hq + it.h) * D;
#pragma unroll
                for (int cc = 0; cc < D / 32; ++cc) {
                    uint32_t o[32];
                    if (nt > 0) {
                        tmem_ld32(tO + cc * 32, o);
                        tmem_wait_ld();
                        if (cc == D / 32 - 1) {   // the accumulator is in registers: the next item may overwrite it
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(bar_o_free(t));
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = 0;
                    }
                    if (alive && row < p.Sq) {
#pragma unroll
                        for (int v4 = 0; v4 < 4; ++v4) {
                            uint4 pk;
                            pk.x = pack_bf16_rn(__uint_as_float(o[v4 * 8 + 0]) * inv, __uint_as_float(o[v4 * 8 + 1]) * inv);
                            pk.y = pack_bf16_rn(__uint_as_float(o[v4 * 8 + 2]) * inv, __uint_as_float(o[v4 * 8 + 3]) * inv);
                            pk.z = pack_bf16_rn(__uint_as_float(o[v4 * 8 + 4]) * inv, __uint_as_float(o[v4 * 8 + 5]) * inv);
                            pk.w = pack_bf16_rn(__uint_as_float(o[v4 * 8 + 6]) * inv, __uint_as_float(o[v4 * 8 + 7]) * inv);
                            *reinterpret_cast<uint4*>(orow + cc * 32 + v4 * 8) = pk;
                        }
                    }
                }
            }
            tiles += nt;
        }
    }

    if (tid == 256) ROWMAX_STAMP(2, 63, 6);
    if constexpr (SPLIT) {
        cluster_arrive();
        cluster_wait();     // nobody reads this CTA's shared memory any more
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 256) ROWMAX_STAMP(2, 63, 7);
#ifdef ROWMAX_TRACE
    if (tid == 0 && p.trace != nullptr && p.trace_block < 0) p.trace[blockIdx.x] = clock64() - trace_t0;   // per-CTA busy time
#endif
    if (warp == 12) {
        __syncwarp();      // the lanes leave the bounded wait on bar_drain each by itself, and this wants the whole warp
        tmem_dealloc(tmem, kTmemCols);
    }
}

// Launches the plain form.
template <int D, int IN, int MODE, bool TAU = false>
static cudaError_t launch_ws(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                             const AttnParams& p, cudaStream_t stream) {
    using W = WsCfg<D, IN == kInFP8>;
    auto kern = attn_fwd_ws_kernel<D, IN, MODE, false, TAU>;
    static bool configured[64] = {};   // per device: the shared-memory opt-in of this instance
    int dev = 0, sm_count = 0;
    cudaError_t e = device_and_sms(&dev, &sm_count);
    if (e != cudaSuccess) return e;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, W::kSmemBytes);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    const long long n_pairs = (p.Sq + 2 * kTileM - 1) / (2 * kTileM);
    const long long items = n_pairs * p.Hq * p.B;
    if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
    // persistent CTAs: one per SM (shared memory and TMEM allow no more), each walking its share of the items
    const unsigned blocks = static_cast<unsigned>(items < sm_count ? items : sm_count);
    // Programmatic dependent launch: the set-up of this kernel (barriers, TMEM, first instructions) overlaps the end of the
    // kernel before it in the stream, 1.1 us (2 heads x 256 keys 8.6 -> 7.4 us, 16 x 1K e4m3 20.3 -> 19.4).  Not where a CTA
    // takes more than one item: CTAs that become resident in the order in which SMs fall free, instead of all at once, run
    // longer there than the overlap saves (48 heads x 2K bf16 60.5 -> 62.6 us).
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = W::kSmemBytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = items <= sm_count ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, tq, tk, tv, p);
}

}  // namespace rowmax
