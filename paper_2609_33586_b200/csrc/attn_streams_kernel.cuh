// Attention forward with one query tile per CTA and two streams of key tiles.
//
// The plain form (attn_fwd_kernel.cuh) keeps its two softmax warpgroups busy with two query tiles that share the staged K/V
// tiles.  Here both work on ONE query tile: key tiles take turns, tile G of the CTA's walk (counted over all its items) belongs
// to stream G mod 2, which has a softmax warpgroup, a score buffer and an O accumulator of its own.
//
// What bounds it: at 16 bits and D = 128 a tile takes 1700 to 2000 clocks, of which the tensor pipe is active in two thirds (nominally
// 1024) and shared memory passes 160 KB (64 KB of K and V in, 96 KB of operands out; 1280 clocks at 128 bytes a clock), the rest
// being hand-offs; elsewhere the chain of one warpgroup, as in the plain form.  A tile
// takes 0.52 to 0.62 of a step of the plain form, which is a tile of two query tiles; so it pays where the plain form's coarser
// items leave SMs idle (streams_pay in plan.h).  In steady streams of calls 16 x 1K e4m3 h15 17.5 -> 14.0 us, 512 queries on 16K
// (32/8 heads, bf16 h15) 200 in the plain and 164 in the split form -> 147, cross attention 36 heads x 1337 x 2803 bf16 exact
// 92.9 -> 83.2 (in short streams, at a higher clock, 143 and 76).  Pairs of CTAs with cta_group::2 and half a K/V tile each were
// no faster (in short streams 16.0, 144 and 78 us against 14.1, 143 and 76): their hand-offs take longer than the operand reads
// that they save.
//
// Semantics are those of the sequential loop: the anchor that tile g starts from is the one tile g - 1 left, handed from
// warpgroup to warpgroup through shared memory as soon as a tile's row maximum is known, half a period before the other needs it.
// So P holds the bits that it has in the plain form.  (The exact modes on 16-bit inputs could do with an anchor for each stream,
// but P would then be rounded about other maxima: O 2e-3 away in the 2-norm instead of 1e-4, for 84.6 us instead of 85.3 in cross
// attention of 36 heads x 1337 x 2803.)  Only the sums are kept per stream and joined at the end: O = (a_0 O_0 + a_1 O_1) dv / l
// with a_t = 2^((m_t - m) c).
//   warpgroup 0/1  softmax of stream 0/1: one thread per row
//   warpgroup 2    correction (rescales the accumulators) and epilogue (joins them and stores O)
//   warp 12        MMA issuer: P V of tile G, then S of tile G + 2, which may be the next item's
//   warp 13        TMA producer: V(G - 2) and K(G) arrive as one pair of ring slots
// TMEM columns: S_0/P_0 [0,128), S_1/P_1 [128,256), O_0 [256,384), O_1 [384,512).
#pragma once
#include "attn_fwd_kernel.cuh"

namespace rowmax {

namespace {

template <int D, bool FP8>
struct StreamsCfg {
    using C = TileCfg<D, FP8>;
    static constexpr int kQBufs = C::kTileBytes <= 16384 ? 2 : 1;        // query tiles staged
    static constexpr int kPairs = C::kTileBytes <= 16384 ? 4 : 3;        // pairs of K/V ring slots
    static constexpr int kQBytes = kQBufs * C::kTileBytes;
    static constexpr int kRingBytes = 2 * kPairs * C::kTileBytes;
    static constexpr int kScaleOff = kQBytes + kRingBytes;       // float alpha[2][128]
    static constexpr int kAnchorOff = kScaleOff + 2 * 128 * 4;   // float anchor[128]: of the last tile that has its maximum
    static constexpr int kFinOff = kAnchorOff + 128 * 4;         // float factor[2][128] of the accumulators (before: m and l of a stream)
    static constexpr int kBarOff = kFinOff + 2 * 128 * 4;
    static constexpr int kNumBars = 2 * kPairs + 16;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;
    static constexpr int kCountOff = kMiscOff + 16;              // int done[4], left[4]: per warp of rows
    static constexpr int kSmemBytes = kCountOff + 32;
    static_assert(kSmemBytes <= 232448, "exceeds the 227 KB shared memory of an sm_100 CTA");
};

// Register split (see the plain form).  The softmax warps have no epilogue here, the MMA warp looks two tiles ahead and the
// correction warps join two accumulators: with 200 / 56 / 56 the MMA warp spills in its loop, with 192 / 64 / 64 only the epilogue
// does (32 bytes, once an item).
constexpr int kStreamRegSoftmax = 192, kStreamRegOther = 64;
static_assert(256 * kStreamRegSoftmax + 256 * kStreamRegOther <= 512 * 128, "setmaxnreg targets exceed the launch allocation");

// One work item: a query tile of one (batch, head) and its key tiles (0: no row sees a key).  Heaviest first, as in the plain form.
struct StreamItem {
    int h, b, hk, q0, n;
};
__device__ __forceinline__ StreamItem decode_stream_item(int w, const AttnParams& p, int n_tiles, int bh) {
    StreamItem it;
    const int rem = w % bh;
    it.q0 = (n_tiles - 1 - w / bh) * kTileM;
    it.h = rem % p.Hq;
    it.b = rem / p.Hq;
    it.hk = it.h / p.group;
    const int kv_end = p.causal ? min(p.Sk, it.q0 + kTileM + p.Sk - p.Sq) : p.Sk;
    it.n = kv_end > 0 ? (kv_end + kTileN - 1) / kTileN : 0;
    return it;
}

// Waits (bounded) until a counter in shared memory has come to `want`.  Counters only grow, so unlike a barrier's phases they
// can be looked at by whoever needs them, however many steps apart.
__device__ __forceinline__ void wait_count(uint32_t at, int want, const WaitCtx& ctx, int code) {
    if (ld_acquire_shared(at) >= want) return;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (ld_acquire_shared(at) >= want || flag_is_set(ctx.cta_abort)) return;
        if (*reinterpret_cast<volatile int*>(ctx.global_status) != 0 || clock64() - t0 > ctx.limit_cycles) {
            write_flag(ctx.cta_abort, 1);
            atomicCAS(ctx.global_status, 0, code);
            return;
        }
    }
}

// Rescaling, masking and weights as in the roles of the plain form, where the same code stands inline: as calls of these functions
// it ran slower there (16K, 32/8 heads, bf16 h15: 1834 -> 1861 us; 48 heads x 2K 64.9 -> 65.4; two runs of one side differ by up to 1 %).

// Multiplies a row of an O accumulator (one row per thread, at the warp's lanes of `tO`) by alpha, unless no row of the warp moves.
template <int D>
__device__ __forceinline__ void rescale_o(uint32_t tO, float alpha) {
    __syncwarp();
    tc_fence_after();
    if (__any_sync(0xffffffffu, alpha != 1.0f)) {
#pragma unroll
        for (int cc = 0; cc < D / 16; ++cc) {
            uint32_t o[16];
            tmem_ld16(tO + cc * 16, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
                const float2 v = fmul2(make_float2(__uint_as_float(o[i]), __uint_as_float(o[i + 1])), make_float2(alpha, alpha));
                o[i] = __float_as_uint(v.x);
                o[i + 1] = __float_as_uint(v.y);
            }
            tmem_st16(tO + cc * 16, o);
        }
        tmem_wait_st();
    }
    tc_fence_before();
}

// Scores at columns >= limit become -inf.
__device__ __forceinline__ void mask_scores(uint32_t (&s)[4][32], int limit) {
#pragma unroll
    for (int cc = 0; cc < 4; ++cc)
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (cc * 32 + i >= limit) s[cc][i] = __float_as_uint(-INFINITY);
}

// The weights of one row of a key tile, its scores in s and its anchor m_use: P goes to TMEM at tP, the row sum is returned.
// LATE: post_alpha is called after the first 32 weights (else not at all).  score_floor bounds the row's scores from below
// (h15 family on fp8 inputs).
template <bool FP8, bool HALF, int MODE, bool LATE, typename PostAlpha>
__device__ __forceinline__ float tile_weights(uint32_t (&s)[4][32], bool masked_tile, int col_limit, float m_use, float score_floor,
                                              const AttnParams& p, uint32_t tP, PostAlpha post_alpha) {
    constexpr int kFam = h15_family_k(MODE);   // h15 family: the map takes the offset times 2^kFam
    const float c_eff = static_cast<float>(1 << kFam) * p.c;
    constexpr float p_off = static_cast<float>(PFormat<FP8, MODE>::kOffLog2);  // log2 of the P / row-sum scale
    // 16-bit inputs: the h15 family uses the saturating form of weights_chunk32 (no row-minimum pass, no
    // clamped or masked variants).  fp8 inputs keep the packed form: there a bound on the key magnitude already
    // removes the row-minimum pass, and the scalar multiply-adds of the saturating form cost more issue slots than
    // they save (in the plain form 4 to 6 %).
    constexpr bool kSatForm = kFam > 0 && !FP8;
    // exact: x = s*c - m*c + P offset;  h15 family: scaled input 2^K x = s*(2^K c) - m*(2^K c);  pot: x = s*c - m*c
    RowScale rs;
    const float nmc = (is_exact_like(MODE) ? p_off : 0.0f) - m_use * c_eff;
    rs.c = make_float2(c_eff, c_eff);
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
            tmem_st16(tP + cc * 16, pw);
        }
    } else if (is_pot(MODE) && masked_tile) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            uint32_t pw[16];
            weights_chunk32<FP8, MODE, true, true, HALF>(s[cc], rs, col_limit - cc * 32, acc, pw);
            if constexpr (FP8) tmem_st8(tP + cc * 8, pw);
            else tmem_st16(tP + cc * 16, pw);
            if (LATE && cc == 0) post_alpha();
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
                if constexpr (FP8) tmem_st8(tP + cc * 8, pw);
                else tmem_st16(tP + cc * 16, pw);
                if (LATE && cc == 0) post_alpha();
            }
        } else {
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                uint32_t pw[16];
                weights_chunk32<FP8, MODE, false, false, HALF>(s[cc], rs, 32, acc, pw);
                if constexpr (FP8) tmem_st8(tP + cc * 8, pw);
                else tmem_st16(tP + cc * 16, pw);
                if (LATE && cc == 0) post_alpha();
            }
        }
    }
    return (acc[0].x + acc[0].y) + (acc[1].x + acc[1].y);
}

// Stores 16 rows x 32 columns of O as bf16.  `v` is laid out as tcgen05.ld.16x256b.x4 gives it: of each 8 columns lane i has
// columns 2 (i mod 4) and the next of row i / 4 (v[4k], v[4k + 1]) and of row i / 4 + 8 (v[4k + 2], v[4k + 3]).  The four lanes of
// a row exchange their words so that each has 16 bytes in a row: a store then takes 8 rows x 64 bytes, whole sectors, where one
// row per thread takes 32 rows x 16 bytes.  (In the plain form, cross attention of 1337 x 2803: 93.9 -> 90.2 us.)
__device__ __forceinline__ void store_rows16(const uint32_t (&v)[16], __nv_bfloat16* base, size_t row_stride, int rows, int lane) {
    const bool odd = lane & 1, upper = lane & 2;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int row = (lane >> 2) + 8 * half;
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = pack_bf16_rn(__uint_as_float(v[4 * k + 2 * half]), __uint_as_float(v[4 * k + 2 * half + 1]));
        // word k of lane j becomes word j of lane k
        const uint32_t x01 = __shfl_xor_sync(0xffffffffu, odd ? w[0] : w[1], 1), x23 = __shfl_xor_sync(0xffffffffu, odd ? w[2] : w[3], 1);
        if (odd) { w[0] = x01; w[2] = x23; }
        else { w[1] = x01; w[3] = x23; }
        const uint32_t y0 = __shfl_xor_sync(0xffffffffu, upper ? w[0] : w[2], 2), y1 = __shfl_xor_sync(0xffffffffu, upper ? w[1] : w[3], 2);
        const uint4 pk = upper ? make_uint4(y0, y1, w[2], w[3]) : make_uint4(w[0], w[1], y0, y1);
        if (row < rows) *reinterpret_cast<uint4*>(base + row * row_stride + 8 * (lane & 3)) = pk;
    }
}

}  // namespace

template <int D, int IN, int MODE>
__global__ void __launch_bounds__(512, 1)
attn_fwd_streams_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
    constexpr bool FP8 = IN == kInFP8;
    constexpr bool HALF = IN == kInFP16;
    using C = TileCfg<D, FP8>;
    using W = StreamsCfg<D, FP8>;
    constexpr int NP = W::kPairs;
    constexpr bool kOutOfStep = FP8 && is_exact_like(MODE);
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sQ = smem_u32(smem);
    const uint32_t sRing = sQ + W::kQBytes;
    const uint32_t sScale = smem_u32(smem + W::kScaleOff);
    const uint32_t sAnchor = smem_u32(smem + W::kAnchorOff);
    const uint32_t sFin = smem_u32(smem + W::kFinOff);
    const uint32_t bar0 = smem_u32(smem + W::kBarOff);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + W::kMiscOff);
    const uint32_t abort_at = smem_u32(smem + W::kMiscOff + 4), leave_at = smem_u32(smem + W::kMiscOff + 8);
    const uint32_t count_done = smem_u32(smem + W::kCountOff), count_left = count_done + 16;
    const WaitCtx wctx{abort_at, p.status, kWaitLimitCycles};

    using Ring = StreamRing<NP>;
    auto bar_kv_full = [&](int pair) { return bar0 + 8u * Ring::bar(pair); };              // TMA -> MMA: V(G - 2) and K(G)
    auto bar_kv_empty = [&](int pair) { return bar0 + 8u * (NP + Ring::bar(pair)); };      // MMA -> TMA
    auto bar_x = [&](int which, int t) { return bar0 + 8u * (2 * NP + 2 * which + t); };
    auto bar_q_full = [&](int b) { return bar_x(0, b); };      // TMA -> MMA: Q of the item landed
    auto bar_q_empty = [&](int b) { return bar_x(1, b); };     // MMA -> TMA: last S MMA of the item done
    auto bar_s_full = [&](int t) { return bar_x(2, t); };      // MMA -> softmax: S(G) is in TMEM
    auto bar_p_full = [&](int t) { return bar_x(3, t); };      // softmax and correction -> MMA: P(G) is in TMEM, O_t rescaled
    auto bar_scale = [&](int t) { return bar_x(4, t); };       // softmax -> correction: alpha(G) in shared memory
    auto bar_anchor = [&](int t) { return bar_x(5, t); };      // softmax -> the other softmax: anchor after tile G
    const uint32_t bar_o_full = bar_x(6, 0);                   // MMA -> epilogue: the last P V of the item accumulated
    const uint32_t bar_o_free = bar_x(6, 1);                   // epilogue -> MMA: both accumulators have been read out
    const uint32_t bar_fin = bar_x(7, 0);                      // softmax -> epilogue: factors of the accumulators
    const uint32_t bar_drain = bar_x(7, 1);                    // the MMA warp's last commit

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wg = warp >> 2;
    if ((smem_u32(smem) & 1023u) != 0) {
        if (tid == 0) atomicCAS(p.status, 0, (kRoleSetup << 8) | kBarAlign);
        return;
    }
    // As in the plain form one thread reads the sticky status word, and the CTA leaves as a whole if it is set.
    if (tid == 0) {
        const int set = *reinterpret_cast<volatile int*>(p.status) != 0 ? 1 : 0;
        write_flag(abort_at, set);
        write_flag(leave_at, set);
    }
    const int n_tiles = (p.Sq + kTileM - 1) / kTileM;
    const int bh = p.Hq * p.B;
    const int n_items = n_tiles * bh;
    const int cta = blockIdx.x, n_ctas = gridDim.x;
    const int shift = p.Sk - p.Sq;

    if (warp == 13) {
        if (lane < NP) {
            mbar_init(bar0 + 8u * lane, 2);            // V(G - 2) and K(G)
            mbar_init(bar0 + 8u * (NP + lane), 1);
        } else if (lane >= 16 && lane < 18) {
            const int t = lane - 16;
            mbar_init(bar_q_full(t), 1);
            mbar_init(bar_q_empty(t), 1);
            mbar_init(bar_s_full(t), 1);
            mbar_init(bar_p_full(t), 8);      // one arrival per softmax warp, one per correction warp
            mbar_init(bar_scale(t), 4);
            mbar_init(bar_anchor(t), 4);
        } else if (lane == 18) {
            mbar_init(bar_o_full, 1);
            mbar_init(bar_o_free, 4);
            mbar_init(bar_fin, 4);
            mbar_init(bar_drain, 1);
        } else if (lane >= 20 && lane < 28) {
            write_flag(count_done + 4 * (lane - 20), 0);
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
    griddep_wait();        // what follows reads the caller's tensors
    griddep_launch();
    if (flag_is_set(leave_at)) {
        if (warp == 12) tmem_dealloc(tmem, kTmemCols);
        return;
    }
    auto get_item = [&](int w) { return decode_stream_item(w, p, n_tiles, bh); };
    auto tmem_S = [&](int t) { return tmem + 128u * t; };
    auto tmem_O = [&](int t) { return tmem + 256u + 128u * t; };

    constexpr uint32_t fmt_16 = HALF ? kFmtF16 : kFmtBF16;
    constexpr uint32_t fmt_ab = FP8 ? kFmtE4M3 : fmt_16;
    constexpr uint32_t fmt_p = FP8 ? (PFormat<FP8, MODE>::kE4M3 ? kFmtE4M3 : kFmtE5M2) : fmt_16;
    constexpr uint32_t idesc_s = umma_idesc(fmt_ab, fmt_ab, false, false, kTileM, kTileN);
    constexpr uint32_t idesc_pv = umma_idesc(fmt_p, fmt_ab, false, true, kTileM, D);
    constexpr float p_off = static_cast<float>(PFormat<FP8, MODE>::kOffLog2);

    if (wg == 3) {
        reg_dec<kStreamRegOther>();
        if (warp == 13 && lane == 0) {
            // ------------------------------------------------------------ TMA producer
            int walked = 0;       // tiles of the walk so far
            int items = 0;        // items with tiles so far
            StreamItem it;
            int v_b[2] = {0, 0}, v_hk[2] = {0, 0}, v_tile[2] = {0, 0};     // the last two tiles, whose V comes with the K of two tiles later
            auto load_tile = [&](const CUtensorMap* tm, uint32_t dst, uint32_t bar, int head, int row0, int b) {
                mbar_arrive_expect_tx(bar, C::kTileBytes);
#pragma unroll
                for (int bx = 0; bx < C::kBoxes; ++bx) tma_load_4d(dst + bx * C::kBoxBytes, tm, bar, bx * C::kBoxElems, head, row0, b);
            };
            int j = 0;
            // After an expired wait nothing more is loaded (see the plain form).
            StreamOps ops{[&](int pair) { mbar_arrive(bar_kv_full(pair)); },
                          [&](int pair) {
                              mbar_wait(bar_kv_empty(pair), Ring::ph_empty(pair), wctx, (kRoleLoad << 8) | kBarKvEmpty);
                              return !flag_is_set(abort_at);
                          },
                          [&](int pair) { load_tile(&tmK, sRing + Ring::slot_k(pair) * C::kTileBytes, bar_kv_full(pair), it.hk, j * kTileN, it.b); },
                          [&](int pair) { load_tile(&tmV, sRing + Ring::slot_v(pair) * C::kTileBytes, bar_kv_full(pair), v_hk[0], v_tile[0] * kTileN, v_b[0]); }};
            bool ok = true;
            for (int round = 0; ok; ++round) {
                const int w = item_index(round, cta, n_ctas);
                if (w >= n_items) break;
                it = get_item(w);
                for (j = 0; j < it.n; ++j) {
                    ok = stream_tile(ops, walked);
                    if (!ok) break;
                    ++walked;
                    v_b[0] = v_b[1]; v_hk[0] = v_hk[1]; v_tile[0] = v_tile[1];
                    v_b[1] = it.b; v_hk[1] = it.hk; v_tile[1] = j;
                    if (j == 0) {
                        const int buf = items % W::kQBufs;
                        mbar_wait(bar_q_empty(buf), ((items / W::kQBufs) & 1) ^ 1, wctx, (kRoleLoad << 8) | kBarQEmpty);
                        ok = !flag_is_set(abort_at);
                        if (!ok) break;
                        load_tile(&tmQ, sQ + buf * C::kTileBytes, bar_q_full(buf), it.h, it.q0, it.b);
                        ++items;
                    }
                }
            }
            // the last two tiles' V
            int pairs = walked;
            for (int e = walked; ok && e < walked + 2; ++e) {
                ok = stream_tail(ops, e);
                if (ok) pairs = e + 1;
                v_b[0] = v_b[1]; v_hk[0] = v_hk[1]; v_tile[0] = v_tile[1];
            }
            // Every load this thread issued has to land before the CTA ends (see the plain form).
            for (int pair = pairs > NP ? pairs - NP : 0; pair < pairs; ++pair)
                if (stream_pair_is_used(pair, walked)) mbar_wait_quiet(bar_kv_full(pair), Ring::ph_full(pair), kDrainLimitCycles);
            for (int i = items > W::kQBufs ? items - W::kQBufs : 0; i < items; ++i)
                mbar_wait_quiet(bar_q_full(i % W::kQBufs), (i / W::kQBufs) & 1, kDrainLimitCycles);
        } else if (warp == 12) {
            // ------------------------------------------------------------ MMA issuer
            const bool leader = elect_one();
            constexpr uint32_t desc_hi = umma_desc_hi_sw(C::kSwizzle);
            const uint32_t q_lo0 = umma_desc_lo(sQ, 16);
            const uint32_t ring_lo_k = umma_desc_lo(sRing, 16);               // K tiles: K-major
            const uint32_t ring_lo_v = umma_desc_lo(sRing, C::kBoxBytes);     // V tiles: MN-major, LBO = next block of columns
            constexpr uint32_t kTileLo = C::kTileBytes >> 4;
            auto issue_s = [&](int t, uint32_t q_lo, uint32_t k_lo) {
#pragma unroll
                for (int ks = 0; ks < C::kQkSteps; ++ks) {
                    const uint32_t off = ((ks / C::kStepsPerBox) * C::kBoxBytes + (ks % C::kStepsPerBox) * 32) >> 4;
                    umma_ss_lo<FP8>(tmem_S(t), q_lo + off, k_lo + off, desc_hi, idesc_s, ks > 0 ? 1u : 0u);
                }
            };
            auto issue_pv = [&](int t, uint32_t v_lo, bool accumulate) {
#pragma unroll
                for (int ks = 0; ks < C::kPvSteps; ++ks) {
                    const uint32_t off = (ks * C::kUmmaK * C::kSwizzle) >> 4;
                    umma_ts_lo<FP8>(tmem_O(t), tmem_S(t) + ks * 8, v_lo + off, desc_hi, idesc_pv, (accumulate || ks > 0) ? 1u : 0u);
                }
            };
            auto tiles_of = [&](int round) {       // of the item of a round, 0 beyond the last
                const int w = item_index(round, cta, n_ctas);
                return w < n_items ? get_item(w).n : 0;
            };
            // The scores run two tiles ahead of the products: tile s_j of s_n of the item that uses Q for the s_item-th time.
            int s_round = 0, s_n = tiles_of(0), s_j = 0, s_item = 0;
            auto wait_pair = [&](int pair) { mbar_wait(bar_kv_full(pair), Ring::ph_full(pair), wctx, (kRoleMma << 8) | kBarKvFull); };
            auto wait_q = [&]() {       // for an item's first scores
                if (s_j == 0 && s_n > 0) mbar_wait(bar_q_full(s_item % W::kQBufs), (s_item / W::kQBufs) & 1, wctx, (kRoleMma << 8) | kBarQFull);
            };
            auto next_s = [&](int G, bool ok) {    // scores of tile G: its K is there, its Q has been waited for
                if (s_n == 0) return;
                const int t = G & 1, buf = s_item % W::kQBufs;
                if (leader) {
                    if (ok) issue_s(t, q_lo0 + buf * kTileLo, ring_lo_k + Ring::slot_k(G) * kTileLo);
                    umma_commit(bar_s_full(t));
                    if (s_j + 1 == s_n) umma_commit(bar_q_empty(buf));
                    umma_commit(bar_kv_empty(G));       // V(G - 2), whose product was issued before, and K(G)
                }
                __syncwarp();
                if (++s_j == s_n) {
                    s_n = tiles_of(++s_round);
                    s_j = 0;
                    ++s_item;
                }
            };
            for (int G = 0; G < 2; ++G)
                if (s_n > 0) {
                    wait_pair(G);
                    wait_q();
                    tc_fence_after();
                    next_s(G, !flag_is_set(abort_at));
                }
            int G = 0, items = 0;
            for (int round = 0;; ++round) {
                const int n = tiles_of(round);
                if (n == 0) break;         // items without key tiles come last
                for (int g = 0; g < n; ++g, ++G) {
                    const int t = G & 1;
                    const bool ok = !flag_is_set(abort_at);
                    wait_pair(G + 2);
                    wait_q();
                    if (g == 0) mbar_wait_poll(bar_o_free, (items & 1) ^ 1, wctx, (kRoleMma << 8) | kBarOFree);
                    mbar_wait_poll(bar_p_full(t), (G >> 1) & 1, wctx, (kRoleMma << 8) | kBarPFull);
                    tc_fence_after();
                    if (leader) {
                        if (ok) issue_pv(t, ring_lo_v + Ring::slot_v(G + 2) * kTileLo, g >= 2);
                        if (g + 1 == n) umma_commit(bar_o_full);
                    }
                    __syncwarp();
                    next_s(G + 2, ok);
                }
                ++items;
            }
            // No MMA of this thread may still be running when TMEM is handed back (see the plain form).
            if (leader) umma_commit(bar_drain);
            mbar_wait_quiet(bar_drain, 0, kDrainLimitCycles);
        }
    } else if (wg == 2) {
        // ---------------------------------------------------------------- correction and epilogue
        reg_dec<kStreamRegOther>();
        // The kernel before this one may have set the status word after the check above: whoever stores looks again, and stores
        // nothing if it is set (the hand-offs go on).
        const bool mute = *reinterpret_cast<volatile int*>(p.status) != 0;
        const int r = tid & 127;
        const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
        int G = 0, items = 0;
        int due = -1, due_first = 0;     // an item whose O waits for its epilogue; the stream of its first tile
        for (int round = 0;; ++round) {
            const int w = item_index(round, cta, n_ctas);
            StreamItem it;
            it.n = 0;
            if (w < n_items) it = get_item(w);
            if (due >= 0) {
                const StreamItem e = get_item(due);
                const int first = due_first;
                float f_first = 0.f, f_second = 0.f;
                if (e.n > 0) {
                    mbar_wait(bar_fin, items & 1, wctx, (kRoleEpi << 8) | kBarFin);
                    f_first = ld_shared_f32(sFin + (first * 128 + r) * 4);
                    if (e.n > 1) f_second = ld_shared_f32(sFin + ((first ^ 1) * 128 + r) * 4);
                    ++items;
                    __syncwarp();
                    if (lane == 0) st_release_shared(count_done + 4 * (warp & 3), items);
                    mbar_wait(bar_o_full, (items - 1) & 1, wctx, (kRoleEpi << 8) | kBarOFull);
                    __syncwarp();
                    tc_fence_after();
                }
                const bool alive = !mute && !flag_is_set(abort_at);      // after an expired wait the accumulators are not to be trusted
                const int warp_row = e.q0 + (warp & 3) * 32;
                const size_t row_stride = static_cast<size_t>(p.Hq) * D;
                __nv_bfloat16* obase = reinterpret_cast<__nv_bfloat16*>(p.o) + ((static_cast<size_t>(e.b) * p.Sq + warp_row) * p.Hq + e.h) * D;
                const int rows = alive ? p.Sq - warp_row : 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int lo = 16 * h + (lane >> 2);
                    const float a_lo = __shfl_sync(0xffffffffu, f_first, lo), a_hi = __shfl_sync(0xffffffffu, f_first, lo + 8);
                    const float b_lo = __shfl_sync(0xffffffffu, f_second, lo), b_hi = __shfl_sync(0xffffffffu, f_second, lo + 8);
#pragma unroll
                    for (int cb = 0; cb < D / 32; ++cb) {
                        uint32_t o[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = 0;
                        if (e.n > 0) {
                            uint32_t o2[16];
                            const uint32_t at = lane_base + (static_cast<uint32_t>(16 * h) << 16) + cb * 32;
                            tmem_ld_16x256b_x4(tmem_O(first) + at, o);
                            if (e.n > 1) tmem_ld_16x256b_x4(tmem_O(first ^ 1) + at, o2);
                            tmem_wait_ld();
                            if (h == 1 && cb == D / 32 - 1) {   // the accumulators are in registers: the next item may overwrite them
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) mbar_arrive(bar_o_free);
                            }
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                float v = __uint_as_float(o[i]) * ((i & 2) ? a_hi : a_lo);
                                if (e.n > 1) v = fmaf(__uint_as_float(o2[i]), (i & 2) ? b_hi : b_lo, v);
                                o[i] = __float_as_uint(v);
                            }
                        }
                        store_rows16(o, obase + 16 * h * row_stride + cb * 32, row_stride, rows - 16 * h, lane);
                    }
                }
                if (alive && e.q0 + r < p.Sq && e.n == 0 && p.lse != nullptr)
                    p.lse[(static_cast<size_t>(e.b) * p.Hq + e.h) * p.Sq + e.q0 + r] = -INFINITY;
            }
            if (w >= n_items) break;
            due = w;
            due_first = G & 1;
            for (int g = 0; g < it.n; ++g, ++G) {
                const int t = G & 1;
                mbar_wait(bar_scale(t), (G >> 1) & 1, wctx, (kRoleCorr << 8) | kBarScale);
                const float alpha = ld_shared_f32(sScale + (t * 128 + r) * 4);
                if (g >= 2) rescale_o<D>(tmem_O(t) + lane_base, alpha);     // P V(G - 2) is complete: alpha(G) was posted after S(G) was seen
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p_full(t));
            }
        }
    } else {
        // ---------------------------------------------------------------- softmax of stream t
        reg_inc<kStreamRegSoftmax>();
        const bool mute = *reinterpret_cast<volatile int*>(p.status) != 0;
        const int t = wg;
        const int r = tid & 127;
        const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_S(t) + lane_base;
        constexpr int kFam = h15_family_k(MODE);
        int base = 0;       // tiles of earlier items
        int items = 0;      // items with key tiles so far
        for (int round = 0;; ++round) {
            const int w = item_index(round, cta, n_ctas);
            if (w >= n_items) break;
            const StreamItem it = get_item(w);
            if (it.n == 0) break;       // these come last and are the epilogue's alone
            const int n = it.n;
            const int row = it.q0 + r;
            const int row_limit = p.causal ? min(p.Sk, row + shift + 1) : p.Sk;          // visible keys of this row
            const int tile_limit = p.causal ? min(p.Sk, it.q0 + shift + 1) : p.Sk;       // first key that some row of the tile cannot see
            const int first = (t ^ base) & 1;       // this stream's first tile of the item
            float m_run = -INFINITY, l_run = 0.f;
            float score_floor = -INFINITY;
            if constexpr (FP8 && kFam > 0) {     // lower bound of the row's scores, as in the plain form
                if (n >= first + 7) {
                    mbar_wait(bar_s_full(t), ((base + first) >> 1) & 1, wctx, (kRoleSoftmax << 8) | kBarSFull);
                    score_floor = -448.0f * 1.02f * abs_sum_e4m3_row<D / 16>(sQ + (items % W::kQBufs) * C::kTileBytes + r * D);
                }
            }
            for (int g = first; g < n; g += 2) {
                const int G = base + g;
                float m_prev = -INFINITY;
                // The anchor after tile G - 1.  Every tile waits for the one before and posts its own, over item boundaries
                // too, so that neither side of the hand-over can get two steps ahead of the other.
                if (G > 0) {
                    mbar_wait(bar_anchor(t ^ 1), ((G - 1) >> 1) & 1, wctx, (kRoleSoftmax << 8) | kBarXmax);
                    if (g > 0) m_prev = ld_shared_f32(sAnchor + r * 4);
                }
                mbar_wait(bar_s_full(t), (G >> 1) & 1, wctx, (kRoleSoftmax << 8) | kBarSFull);
                __syncwarp();
                tc_fence_after();
                uint32_t s[4][32];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) tmem_ld32(tS + cc * 32, s[cc]);
                tmem_wait_ld();
                const bool masked_tile = (g + 1) * kTileN > tile_limit;
                const int col_limit = row_limit - g * kTileN;
                if (masked_tile) mask_scores(s, col_limit);
                const float m_new = fmaxf(m_prev, row_max128(s));
                st_shared_f32(sAnchor + r * 4, m_new);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_anchor(t));
                const float m_use = (m_new == -INFINITY) ? 0.f : m_new;
                const float alpha = ex2_approx((m_run - m_use) * p.c);
                m_run = m_new;
                auto post_alpha = [&]() {
                    st_shared_f32(sScale + (t * 128 + r) * 4, alpha);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_scale(t));
                };
                if constexpr (!kOutOfStep) post_alpha();
                const float l_tile = tile_weights<FP8, HALF, MODE, kOutOfStep>(s, masked_tile, col_limit, m_use, score_floor, p, tS, post_alpha);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p_full(t));
                l_run = l_run * alpha + l_tile;
            }
            // The streams meet: the one that does not have the last tile leaves its anchor and row sum, the other joins them,
            // stores LSE and leaves the factors of the two accumulators for the epilogue.  A row's threads are in the same warp
            // of each warpgroup, so each warp deals with its counterparts alone.
            const bool has_last = ((base + n - 1) & 1) == t;
            if (has_last ? n == 1 : n > 1)
                wait_count(count_done + 4 * (warp & 3), items, wctx, (kRoleSoftmax << 8) | kBarOFree);    // the factors before have been read
            if (!has_last && n > 1) {
                st_shared_f32(sFin + r * 4, m_run);
                st_shared_f32(sFin + (128 + r) * 4, l_run);
                __syncwarp();
                if (lane == 0) st_release_shared(count_left + 4 * (warp & 3), items + 1);
            }
            if (has_last) {
                float m_other = -INFINITY, l_other = 0.f;
                if (n > 1) {
                    wait_count(count_left + 4 * (warp & 3), items + 1, wctx, (kRoleSoftmax << 8) | kBarPart);
                    m_other = ld_shared_f32(sFin + r * 4);
                    l_other = ld_shared_f32(sFin + (128 + r) * 4);
                }
                const float m = fmaxf(m_run, m_other), m_use = m == -INFINITY ? 0.f : m;
                const float a_own = ex2_approx((m_run - m_use) * p.c), a_other = ex2_approx((m_other - m_use) * p.c);
                const float l = n > 1 ? a_own * l_run + a_other * l_other : l_run;
                const bool has_keys = m != -INFINITY && l > 0.f;
                const float inv = has_keys ? p.v_descale / l : 0.f;
                st_shared_f32(sFin + (t * 128 + r) * 4, a_own * inv);
                if (n > 1) st_shared_f32(sFin + ((t ^ 1) * 128 + r) * 4, a_other * inv);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_fin);
                if (row < p.Sq && p.lse != nullptr && !mute && !flag_is_set(abort_at))
                    p.lse[(static_cast<size_t>(it.b) * p.Hq + it.h) * p.Sq + row] =
                        has_keys ? 0.6931471805599453f * (m * p.c + log2f(l) - p_off) : -INFINITY;
            }
            ++items;
            base += n;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 12) {
        __syncwarp();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace rowmax
