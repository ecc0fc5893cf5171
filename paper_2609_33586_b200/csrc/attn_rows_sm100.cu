// Attention forward for few query rows against a long context (decoding, short chunks of new queries).
//
// What bounds this path is reading K and V once.  The query rows of all heads that share a key/value head are packed
// into one tile of N rows (N = 16, 32 or 64), and the matrix products are transposed so that their large side is M:
//     S^T (128 keys x N rows) = K_tile Q^T,          O^T (D x N rows) += V_tile^T P^T,
// both with the K or V tile, as TMA lands it in shared memory, as the first operand.  A cluster of CTAs shares one
// (batch, key/value head): every CTA takes a contiguous share of the key tiles, and the shares meet through
// distributed shared memory, so that there is neither scratch memory nor a second kernel.
//
// The result is that of the sequential loop over key tiles (Sec. 5.2; App. B.1), whose anchor for key tile j is the
// maximum over tiles 0..j: the scores of a CTA's whole share stay in TMEM (512 / N tiles) while the CTAs exchange
// their row maxima, and only then are weights formed, each tile with the anchor that the loop would have had there.
// A context longer than the cluster's TMEM is taken in rounds.  K and V are read exactly once; the ring of
// shared-memory slots goes on filling with V tiles during the exchange.
//
// Per CTA: warps 0-3 softmax (thread = key on the way in, = output dimension on the way out), warp 4 TMA producer,
// warp 5 MMA issuer.  O is accumulated in registers: P V of a tile overwrites the TMEM columns of that tile's scores,
// and each thread adds it to its running sum scaled by the tile's rescale factor.
#include "plan.h"
#include "softmax_math.cuh"

namespace rowmax {

namespace {

constexpr int kRowsThreads = 192;
constexpr int kMaxSlots = 24;
constexpr int kTmemBlockCols = 512;      // floats of the per-(tile, row) arrays: tiles x N <= 512

// Shared-memory layout of one CTA (byte offsets from a 1024-byte boundary; the ring comes first).
template <int D, bool FP8, int N>
struct RowsCfg {
    using C = TileCfg<D, FP8>;
    static constexpr int kQBytes = N * D * C::kElem;
    static constexpr int kQBoxBytes = N * C::kSwizzle;
    static constexpr int kPRowBytes = kTileN * C::kElem;        // 128 (fp8) or 256 bytes of P per query row
    static constexpr int kPBoxBytes = N * 128;
    static constexpr int kPBytes = N * kPRowBytes;              // one of two P buffers
    static constexpr int kArr = kTmemBlockCols * 4;
    // offsets behind the ring
    static constexpr int kQOff = 0;
    static constexpr int kPOff = kQOff + kQBytes;
    static constexpr int kWmaxOff = kPOff + 2 * kPBytes;        // float[4 warps][tile][row]: per-warp tile maxima
    static constexpr int kAnchorOff = kWmaxOff + 4 * kArr;      // float[tile][row]: anchor of the tile
    static constexpr int kAlphaOff = kAnchorOff + kArr;         // float[tile][row]: rescale factor before the tile
    static constexpr int kXmaxOff = kAlphaOff + kArr;           // float[2][CTA][row]: exchanged share maxima
    static constexpr int kLimOff = kXmaxOff + 2 * kMaxCluster * N * 4;   // int[row]: visible keys
    static constexpr int kFacOff = kLimOff + N * 4;             // float[row]: factor to the final anchor
    static constexpr int kMfinOff = kFacOff + N * 4;            // float[row]: final anchor
    static constexpr int kLwOff = kMfinOff + N * 4;             // float[4 warps][row]: row sums
    static constexpr int kLOff = kLwOff + 4 * N * 4;            // float[row]: scaled row sum of this CTA
    static constexpr int kBarOff = kLOff + N * 4;
    static constexpr int kNumBars = 2 * kMaxSlots + kTmemBlockCols / N + 2 + 2 + 1 + 1;
    static constexpr int kMiscOff = kBarOff + kNumBars * 8;     // TMEM address, abort flag
    static constexpr int kFixedBytes = kMiscOff + 16 + 1024;    // + alignment slack
    static_assert(kQBytes % 1024 == 0 && kPBytes % 1024 == 0, "operand tiles start on a swizzle atom");
    static_assert(kMaxSlots <= 31, "one lane per slot sets up the ring's barriers");
};

// Query rows that the softmax warps take at a time: work is skipped in these steps (rows up to the next multiple are
// computed on zero queries and never stored).
template <int N> constexpr int kRowGroup = N == 16 ? 4 : 8;

// TMEM columns of a CTA.  Two CTAs share an SM where the row tile leaves room for two in shared memory: each of them waits
// for hand-offs most of the time (4 x 16K context, e4m3, D = 64: 22 us against 32 us with one; the others 3 to 20 %
// faster or equal). 
template <int N> constexpr int kRowsCols = N == 64 ? 512 : 256;

template <int MODE> struct ModeTag { static constexpr int value = MODE; };

struct RowsParams {
    int cs;           // CTAs per cluster
    int nt;           // key tiles
    int rounds;       // rounds of the cluster over the context
    int share;        // key tiles of one CTA in one round, share * N <= kRowsCols<N>
    int slots;        // ring slots
    int rows;         // Sq * group
    int mode;
};

// barrier ids in status codes of this kernel
enum RowsBar : int { kBarFull = 0x10, kBarBlk = 0x11, kBarP = 0x12, kBarXchg = 0x13, kBarRound = 0x14, kBarSlot = 0x15 };

// Reduces N values per lane over the 32 lanes of a warp (N = 32, 64) in N - 2 or N - 1 exchanges: every step halves the rows
// that a lane keeps.  Lane q ends with rows q * N / 32 .. in v[0 .. N / 32).
template <int N, typename Op>
__device__ __forceinline__ void reduce_scatter_rows(float (&v)[N], int lane, Op op) {
#pragma unroll
    for (int step = 0; step < 5; ++step) {
        const int bit = 16 >> step, cnt = N >> (step + 1);
        const bool upper = (lane & bit) != 0;
#pragma unroll
        for (int j = 0; j < cnt; ++j) {
            const float send = upper ? v[j] : v[j + cnt];
            const float keep = upper ? v[j + cnt] : v[j];
            v[j] = op(keep, __shfl_xor_sync(0xffffffffu, send, bit));
        }
    }
}

// One key (this thread's) of one key tile: the N scores `s` become weights with the anchors of their rows, go into the row
// sums `l` (rescaled by the tile's factors) and, in the format of P, into the operand tile at `pb`.
template <bool FP8, bool HALF, int MODE, int N>
__device__ __forceinline__ void rows_tile_weights(const uint32_t* s, const float* anchor, const float* alpha, float* l,
                                                  int R, bool masked, int key, const int* limits, const AttnParams& p,
                                                  uint8_t* pb, int kl) {
    constexpr int kFam = h15_family_k(MODE);
    constexpr bool kSat = kFam > 0 && !FP8;
    constexpr int kElem = FP8 ? 1 : 2;
    constexpr int kPBoxBytes = N * 128;
    constexpr int G = kRowGroup<N>;
    const float c_eff = static_cast<float>(1 << kFam) * p.c;
    constexpr float p_off = is_exact_like(MODE) ? static_cast<float>(PFormat<FP8, MODE>::kOffLog2) : 0.0f;
    RowScale rs;
    rs.c = make_float2(c_eff, c_eff);
    rs.two22 = p.two22;
    rs.pot_neg_cap = p.pot_neg_cap;
    rs.pot_drop_x = p.pot_drop_x;
    rs.clamp_lo = 0.f;
    if constexpr (kFam > 0) rs.clamp_lo = masked ? h15_clamp_zero<kFam>() : h15_clamp_floor<kFam>();
    constexpr float kR = 126.0f * (1 << kFam), kRm = 127.0f * (1 << kFam);
    const float inv_r = masked ? 1.0f / kRm : 1.0f / kR;
    rs.su = -c_eff * inv_r;
    rs.sat_mul = masked ? -kRm : -kR;
    const int kb = kl * kElem, in_box = kb & 127;
    uint8_t* dst = pb + (kb >> 7) * kPBoxBytes + (in_box & 15);
    const int chunk = in_box >> 4;
    // Groups of rows: all loads, then all weights, then all stores of a group, so that the pairs of a group overlap
    // (byte stores may alias the anchors: pair by pair, every pair waited for the one before, 200 clocks each).
#pragma unroll
    for (int r0 = 0; r0 < N; r0 += G) {
        if (r0 < R) {
            float2 m[G / 2], al[G / 2];
            uint32_t v[G / 2];
#pragma unroll
            for (int i = 0; i < G / 2; i += 2) {
                const float4 m4 = *reinterpret_cast<const float4*>(anchor + r0 + 2 * i);   // 0 stands for "no key yet"
                const float4 a4 = *reinterpret_cast<const float4*>(alpha + r0 + 2 * i);
                m[i] = make_float2(m4.x, m4.y);
                m[i + 1] = make_float2(m4.z, m4.w);
                al[i] = make_float2(a4.x, a4.y);
                al[i + 1] = make_float2(a4.z, a4.w);
            }
#pragma unroll
            for (int i = 0; i < G / 2; ++i) {
                const int r = r0 + 2 * i;
                const float2 mc = fmul2(m[i], make_float2(c_eff, c_eff));
                rs.nmc = make_float2(p_off - mc.x, p_off - mc.y);
                rs.ou = make_float2(mc.x * inv_r, mc.y * inv_r);
                float2 w = weight_pair<FP8, MODE, true, kSat>(make_float2(__uint_as_float(s[r]), __uint_as_float(s[r + 1])), rs, i);
                if constexpr (is_pot(MODE)) {
                    if (masked) {
                        if (key >= limits[r]) w.x = 0.f;
                        if (key >= limits[r + 1]) w.y = 0.f;
                    }
                }
                l[r] = fmaf(l[r], al[i].x, w.x);
                l[r + 1] = fmaf(l[r + 1], al[i].y, w.y);
                if constexpr (FP8) {
                    if constexpr (PFormat<FP8, MODE>::kE4M3) v[i] = __byte_perm(pack_e4m3x2(w.x, w.y), 0u, 0x4140);
                    else v[i] = pack_f16x2_rn(w.x, w.y) >> 8;   // e5m2 is the upper byte of the fp16 pattern, exact for these weights
                } else {
                    if constexpr (HALF) v[i] = pack_f16x2_rn(w.x, w.y);
                    else if constexpr (is_exact_like(MODE)) v[i] = pack_bf16_rn(w.x, w.y);
                    else v[i] = __byte_perm(__float_as_uint(w.x), __float_as_uint(w.y), 0x7632);
                }
            }
#pragma unroll
            for (int i = 0; i < G / 2; ++i) {
                const int r = r0 + 2 * i;
                uint8_t* d0 = dst + r * 128 + ((chunk ^ (r & 7)) << 4);
                uint8_t* d1 = dst + (r + 1) * 128 + ((chunk ^ ((r + 1) & 7)) << 4);
                if constexpr (FP8) {
                    *d0 = static_cast<uint8_t>(v[i]);
                    *d1 = static_cast<uint8_t>(v[i] >> 16);
                } else {
                    *reinterpret_cast<uint16_t*>(d0) = static_cast<uint16_t>(v[i]);
                    *reinterpret_cast<uint16_t*>(d1) = static_cast<uint16_t>(v[i] >> 16);
                }
            }
        }
    }
}

}  // namespace

template <int D, int IN, int N>
__global__ void __launch_bounds__(kRowsThreads, N == 64 ? 1 : 2)
attn_rows_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const void* qptr,
                 const AttnParams p, const RowsParams rp) {
    constexpr bool FP8 = IN == kInFP8;
    constexpr bool HALF = IN == kInFP16;
    using C = TileCfg<D, FP8>;
    using W = RowsCfg<D, FP8, N>;
    constexpr int G = kRowGroup<N>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* fix = ring + rp.slots * C::kTileBytes;
    const uint32_t sRing = smem_u32(ring), sFix = smem_u32(fix);
    float* wmax = reinterpret_cast<float*>(fix + W::kWmaxOff);
    float* anchors = reinterpret_cast<float*>(fix + W::kAnchorOff);
    float* alphas = reinterpret_cast<float*>(fix + W::kAlphaOff);
    int* limits = reinterpret_cast<int*>(fix + W::kLimOff);
    float* fac = reinterpret_cast<float*>(fix + W::kFacOff);
    float* mfin = reinterpret_cast<float*>(fix + W::kMfinOff);
    float* lw = reinterpret_cast<float*>(fix + W::kLwOff);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fix + W::kMiscOff);
    const uint32_t abort_at = smem_u32(fix + W::kMiscOff + 4);
    const WaitCtx wctx{abort_at, p.status, kWaitLimitCycles};
    const uint32_t bar0 = sFix + W::kBarOff;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };                      // TMA -> MMA: slot landed
    auto bar_empty = [&](int s) { return bar0 + 8u * (kMaxSlots + s); };       // MMA -> TMA: slot read
    auto bar_blk = [&](int i) { return bar0 + 8u * (2 * kMaxSlots + i); };     // MMA -> softmax: block i holds S, then P V
    constexpr int kB = 2 * kMaxSlots + kTmemBlockCols / N;
    auto bar_p = [&](int b) { return bar0 + 8u * (kB + b); };                  // softmax -> MMA: P buffer b written
    auto bar_x = [&](int b) { return bar0 + 8u * (kB + 2 + b); };              // share maxima of all CTAs are here
    const uint32_t bar_round = bar0 + 8u * (kB + 4);                           // softmax -> MMA: TMEM blocks free again
    const uint32_t bar_drain = bar0 + 8u * (kB + 5);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = static_cast<int>(cluster_ctarank()), cs = rp.cs;
    const int grp = blockIdx.x / cs;
    const int hk = grp % p.Hkv, b = grp / p.Hkv;
    const int R = rp.rows;

    // key tiles of this CTA in round c: [first, first + count)
    auto first_tile = [&](int c) { return (c * cs + rank) * rp.share; };
    auto tile_count = [&](int c) { return max(0, min(rp.share, rp.nt - first_tile(c))); };

    int loaded = 0;       // producer lane: tiles loaded so far
    auto load_tile = [&](int t0, int i, int n) {   // the i-th tile of a round: K tiles first, then the V tiles
        const int slot = loaded % rp.slots;
        const CUtensorMap* tm = i < n ? &tmK : &tmV;
        const int row0 = (t0 + (i < n ? i : i - n)) * kTileN;
        mbar_arrive_expect_tx(bar_full(slot), C::kTileBytes);
#pragma unroll
        for (int bx = 0; bx < C::kBoxes; ++bx)
            tma_load_4d(sRing + slot * C::kTileBytes + bx * C::kBoxBytes, tm, bar_full(slot), bx * C::kBoxElems, hk, row0, b);
        ++loaded;
    };

    if (warp == 4) {
        // the producer sets up the barriers of its ring and fills it before the rest of the CTA is ready
        if (lane < rp.slots) {
            mbar_init(bar_full(lane), 1);
            mbar_init(bar_empty(lane), 1);
        }
        if (lane == 31) write_flag(abort_at, 0);
        fence_mbar_init();
        __syncwarp();
        griddep_wait();    // what follows reads the caller's tensors
        if (lane == 0) {
            const int t0 = first_tile(0), n = tile_count(0);
            for (int i = 0; i < 2 * n && i < rp.slots; ++i) load_tile(t0, i, n);
        }
        __syncwarp();
    } else if (warp == 5) {
        for (int i = lane; i < kTmemBlockCols / N; i += 32) mbar_init(bar_blk(i), 1);
        if (lane < 2) {
            mbar_init(bar_p(lane), 4);           // one arrival per softmax warp
            mbar_init(bar_x(lane), 4 * cs);      // one arrival per softmax warp of every CTA
        }
        if (lane == 2) mbar_init(bar_round, 4);
        if (lane == 3) mbar_init(bar_drain, 1);
        fence_mbar_init();
        __syncwarp();
        tmem_alloc(smem_u32(tmem_slot), kRowsCols<N>);
        tmem_relinquish();
    } else {
        for (int e = tid; e < 2 * kTmemBlockCols; e += 128) anchors[e] = 0.f;   // and alphas, which follow: rows beyond R stay finite
        for (int r = tid; r < N; r += 128) {
            int lim = p.Sk;
            if (p.causal && r < R) lim = min(p.Sk, r / p.group + 1 + p.Sk - p.Sq);
            limits[r] = lim;
        }
        griddep_wait();
        // Q rows (query qi, head of the group) into the K-major operand tile, swizzled as TMA would have done it
        constexpr int kChunks = D * C::kElem / 16;              // 16-byte pieces of a row
        constexpr int kBoxChunks = C::kSwizzle / 16;
        for (int e = tid; e < N * kChunks; e += 128) {
            const int r = e / kChunks, ch = e % kChunks;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (r < R) {
                const int qi = r / p.group, h = hk * p.group + r % p.group;
                const size_t row = (static_cast<size_t>(b) * p.Sq + qi) * p.Hq + h;
                v = *reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(qptr) + row * (D * C::kElem) + ch * 16);
            }
            const int c = ch % kBoxChunks;
            const int sw = C::kSwizzle == 128 ? (c ^ (r & 7)) : (c ^ ((r >> 1) & 3));
            *reinterpret_cast<uint4*>(fix + W::kQOff + (ch / kBoxChunks) * W::kQBoxBytes + r * C::kSwizzle + sw * 16) = v;
        }
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    griddep_wait();
    griddep_launch();
    // The status word is sticky: while it is set every wait ends soon and nothing is stored.  All CTAs of the
    // cluster still take every step, because the others read their shared memory.
    if (tid == 0 && *reinterpret_cast<volatile int*>(p.status) != 0) write_flag(abort_at, 1);
    cluster_arrive();       // barriers are initialised; waited for before the first remote access and at the end
    const uint32_t tmem = *tmem_slot;

    float l[N], o[N];

    if (warp == 4) {
        if (lane == 0) {
            // ------------------------------------------------------------ TMA producer
            const int filled = loaded;
            int at = 0;           // tiles of the stream passed so far
            for (int c = 0; c < rp.rounds; ++c) {
                const int t0 = first_tile(c), n = tile_count(c);
                for (int i = 0; i < 2 * n && !flag_is_set(abort_at); ++i, ++at) {
                    if (at < filled) continue;
                    mbar_wait_poll(bar_empty(loaded % rp.slots), ((loaded / rp.slots) & 1) ^ 1, wctx, (kRoleLoad << 8) | kBarSlot);
                    if (flag_is_set(abort_at)) break;
                    load_tile(t0, i, n);
                }
            }
            // every copy must have landed before the CTA ends (see attn_fwd_ws_kernel)
            for (int k = loaded > rp.slots ? loaded - rp.slots : 0; k < loaded; ++k)
                mbar_wait_quiet(bar_full(k % rp.slots), (k / rp.slots) & 1, kDrainLimitCycles);
        }
        __syncwarp();
    } else if (warp == 5) {
        // ---------------------------------------------------------------- MMA issuer
        const bool leader = elect_one();
        constexpr uint32_t fmt_ab = FP8 ? kFmtE4M3 : (HALF ? kFmtF16 : kFmtBF16);
        const bool p_e4m3 = is_exact_like(rp.mode) || rp.mode == kH15K3;
        const uint32_t fmt_p = FP8 ? (p_e4m3 ? kFmtE4M3 : kFmtE5M2) : fmt_ab;
        constexpr uint32_t idesc_s = umma_idesc(fmt_ab, fmt_ab, false, false, 128, N);
        const uint32_t idesc_pv = umma_idesc(fmt_ab, fmt_p, true, false, 128, N);
        constexpr uint32_t hi_kv = umma_desc_hi_sw(C::kSwizzle);
        constexpr uint32_t hi_p = umma_desc_hi_sw(128);
        const uint32_t q_lo = umma_desc_lo(sFix + W::kQOff, 16);
        const uint32_t p_lo = umma_desc_lo(sFix + W::kPOff, 16);
        const uint32_t k_lo0 = umma_desc_lo(sRing, 16);
        // V^T as the M-major first operand with M = 128.  For D = 64 the upper 64 rows come from whatever lies one
        // box further (inside this CTA's shared memory); their results are in TMEM lanes that nobody reads.
        const uint32_t v_lo0 = umma_desc_lo(sRing, C::kBoxBytes);
        constexpr uint32_t kTileLo = C::kTileBytes >> 4;
        int idx = 0, np = 0;
        for (int c = 0; c < rp.rounds; ++c) {
            const int n = tile_count(c);
            if (c > 0) mbar_wait_poll(bar_round, (c - 1) & 1, wctx, (kRoleMma << 8) | kBarRound);
            for (int i = 0; i < n; ++i, ++idx) {
                const int slot = idx % rp.slots;
                mbar_wait_poll(bar_full(slot), (idx / rp.slots) & 1, wctx, (kRoleMma << 8) | kBarFull);
                tc_fence_after();
                if (leader) {
                    if (!flag_is_set(abort_at)) {
                        const uint32_t k_lo = k_lo0 + slot * kTileLo;
#pragma unroll
                        for (int ks = 0; ks < C::kQkSteps; ++ks) {
                            const int bx = ks / C::kStepsPerBox, in = (ks % C::kStepsPerBox) * 32;
                            umma_ss_lo2<FP8>(tmem + i * N, k_lo + ((bx * C::kBoxBytes + in) >> 4), hi_kv,
                                             q_lo + ((bx * W::kQBoxBytes + in) >> 4), hi_kv, idesc_s, ks > 0 ? 1u : 0u);
                        }
                    }
                    umma_commit(bar_empty(slot));
                    umma_commit(bar_blk(i));
                }
                __syncwarp();
            }
            for (int i = 0; i < n; ++i, ++idx, ++np) {
                const int slot = idx % rp.slots, buf = np & 1;
                mbar_wait_poll(bar_full(slot), (idx / rp.slots) & 1, wctx, (kRoleMma << 8) | kBarFull);
                mbar_wait_poll(bar_p(buf), (np >> 1) & 1, wctx, (kRoleMma << 8) | kBarP);
                tc_fence_after();
                if (leader) {
                    if (!flag_is_set(abort_at)) {
                        const uint32_t v_lo = v_lo0 + slot * kTileLo;
                        const uint32_t pb_lo = p_lo + buf * (W::kPBytes >> 4);
#pragma unroll
                        for (int ks = 0; ks < C::kPvSteps; ++ks)
                            umma_ss_lo2<FP8>(tmem + i * N, v_lo + ((ks * C::kUmmaK * C::kSwizzle) >> 4), hi_kv,
                                             pb_lo + (((ks / 4) * W::kPBoxBytes + (ks % 4) * 32) >> 4), hi_p, idesc_pv,
                                             ks > 0 ? 1u : 0u);
                    }
                    umma_commit(bar_blk(i));
                    umma_commit(bar_empty(slot));
                }
                __syncwarp();
            }
        }
        if (leader) umma_commit(bar_drain);
        mbar_wait_quiet(bar_drain, 0, kDrainLimitCycles);
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- softmax
        const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
        const int kl = warp * 32 + lane;      // key of a tile on the way in, output dimension on the way out
        constexpr int kRowsPerWarp = N / 4;   // rows whose maxima this warp scans: warp, warp + 4, ...
        constexpr int kBlocks = kTmemBlockCols / N;
        float carry[kRowsPerWarp], own[kRowsPerWarp];   // maximum over all earlier rounds; anchor of l and o
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k) carry[k] = own[k] = -INFINITY;
#pragma unroll
        for (int r = 0; r < N; ++r) l[r] = o[r] = 0.f;
        const int min_limit = limits[0];      // rows are ordered by query: the first sees the fewest keys
        auto load_block = [&](int i, uint32_t (&s)[N]) {
            const uint32_t a = tmem + lane_base + i * N;
            if constexpr (N == 16) {
                tmem_ld16(a, s);
            } else {
#pragma unroll
                for (int cc = 0; cc < N / 32; ++cc) tmem_ld32(a + cc * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[cc * 32]));
            }
            tmem_wait_ld();
        };
        auto mask_scores = [&](uint32_t (&s)[N], int key) {
#pragma unroll
            for (int r = 0; r < N; ++r)
                if (r < R && key >= limits[r]) s[r] = __float_as_uint(-INFINITY);
        };
        int np = 0;
        for (int c = 0; c < rp.rounds; ++c) {
            const int t0 = first_tile(c), n = tile_count(c);
            // row maxima of every tile of the share
            for (int i = 0; i < n; ++i) {
                uint32_t s[N];
                mbar_wait_poll(bar_blk(i), 0, wctx, (kRoleSoftmax << 8) | kBarBlk);
                __syncwarp();
                tc_fence_after();
                load_block(i, s);
                if ((t0 + i + 1) * kTileN > min_limit) mask_scores(s, (t0 + i) * kTileN + kl);
                float* wm = wmax + warp * kTmemBlockCols + i * N;
                if constexpr (N == 16) {
                    float mine = 0.f;
#pragma unroll
                    for (int r0 = 0; r0 < N; r0 += G) {
                        if (r0 < R) {
                            float v[G];
#pragma unroll
                            for (int r = 0; r < G; ++r) v[r] = redux_max(__uint_as_float(s[r0 + r]));
#pragma unroll
                            for (int r = 0; r < G; ++r)
                                if (lane == r0 + r) mine = v[r];
                        }
                    }
                    if (lane < R) wm[lane] = mine;
                } else {
                    float v[N];
#pragma unroll
                    for (int r = 0; r < N; ++r) v[r] = __uint_as_float(s[r]);
                    reduce_scatter_rows<N>(v, lane, [](float x, float y) { return fmaxf(x, y); });
#pragma unroll
                    for (int q = 0; q < N / 32; ++q) wm[lane * (N / 32) + q] = v[q];
                }
            }
            named_barrier<1>(128);
            // running maximum over the share's tiles, per row: one lane per tile
            float pre[kRowsPerWarp];
#pragma unroll
            for (int k = 0; k < kRowsPerWarp; ++k) {
                const int r = warp + 4 * k;
                pre[k] = -INFINITY;
                if (r < R && lane < n) {
                    const float* wm = wmax + lane * N + r;
                    pre[k] = fmaxf(max3(wm[0], wm[kTmemBlockCols], wm[2 * kTmemBlockCols]), wm[3 * kTmemBlockCols]);
                }
            }
#pragma unroll
            for (int d = 1; d < kBlocks; d <<= 1) {
                float u[kRowsPerWarp];
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k) u[k] = __shfl_up_sync(0xffffffffu, pre[k], d);
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k)
                    if (lane >= d) pre[k] = fmaxf(pre[k], u[k]);
            }
            if (c == 0) cluster_wait();   // every CTA has initialised its barriers
#pragma unroll
            for (int k = 0; k < kRowsPerWarp; ++k) {
                const int r = warp + 4 * k;
                const float total = __shfl_sync(0xffffffffu, pre[k], kBlocks - 1);
                if (r < R && lane < cs)
                    st_cluster_f32(mapa(sFix + W::kXmaxOff + (((c & 1) * kMaxCluster + rank) * N + r) * 4, lane), total);
            }
            // Two barriers in turn: a CTA posts round c + 2 only after everybody has read round c.
            if (lane < cs) mbar_arrive_cluster(mapa(bar_x(c & 1), lane));
            mbar_wait_cluster(bar_x(c & 1), (c >> 1) & 1, wctx, (kRoleSoftmax << 8) | kBarXchg);
            __syncwarp();
            {
                float x[kRowsPerWarp], m[kRowsPerWarp];
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k) {
                    const int r = warp + 4 * k;
                    x[k] = -INFINITY;
                    if (lane < cs && r < R)
                        x[k] = *reinterpret_cast<const volatile float*>(fix + W::kXmaxOff + (((c & 1) * kMaxCluster + lane) * N + r) * 4);
                }
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k) m[k] = fmaxf(carry[k], redux_max(lane < rank ? x[k] : -INFINITY));
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k) {
                    carry[k] = fmaxf(carry[k], redux_max(x[k]));
                    m[k] = fmaxf(m[k], pre[k]);          // the anchor of tile `lane`
                }
#pragma unroll
                for (int k = 0; k < kRowsPerWarp; ++k) {
                    const int r = warp + 4 * k;
                    float prev = __shfl_up_sync(0xffffffffu, m[k], 1);
                    if (lane == 0) prev = own[k];
                    const float m_use = m[k] == -INFINITY ? 0.f : m[k];
                    if (lane < n && r < R) {
                        anchors[lane * N + r] = m_use;
                        alphas[lane * N + r] = ex2_approx((prev - m_use) * p.c);
                    }
                }
                if (n > 0) {
#pragma unroll
                    for (int k = 0; k < kRowsPerWarp; ++k) own[k] = __shfl_sync(0xffffffffu, m[k], n - 1);
                }
            }
            named_barrier<1>(128);
            // weights and P V, tile by tile; the product of tile i - 1 is added while tile i's runs
            auto add_product = [&](int i) {
                uint32_t s[N];
                mbar_wait_poll(bar_blk(i), 1, wctx, (kRoleSoftmax << 8) | kBarBlk);
                __syncwarp();
                tc_fence_after();
                load_block(i, s);
#pragma unroll
                for (int r0 = 0; r0 < N; r0 += G) {
                    if (r0 < R) {
#pragma unroll
                        for (int r = r0; r < r0 + G; r += 4) {
                            const float4 al = *reinterpret_cast<const float4*>(alphas + i * N + r);
                            o[r] = fmaf(o[r], al.x, __uint_as_float(s[r]));
                            o[r + 1] = fmaf(o[r + 1], al.y, __uint_as_float(s[r + 1]));
                            o[r + 2] = fmaf(o[r + 2], al.z, __uint_as_float(s[r + 2]));
                            o[r + 3] = fmaf(o[r + 3], al.w, __uint_as_float(s[r + 3]));
                        }
                    }
                }
            };
            auto weigh_share = [&](auto mode) {
                for (int i = 0; i < n; ++i, ++np) {
                    uint32_t s[N];
                    load_block(i, s);
                    const int key = (t0 + i) * kTileN + kl;
                    const bool masked = (t0 + i + 1) * kTileN > min_limit;
                    if (masked) mask_scores(s, key);
                    rows_tile_weights<FP8, HALF, decltype(mode)::value, N>(s, anchors + i * N, alphas + i * N, l, R, masked, key,
                                                                           limits, p, fix + W::kPOff + (np & 1) * W::kPBytes, kl);
                    fence_proxy_async();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_p(np & 1));
                    if (i > 0) add_product(i - 1);
                }
            };
            switch (rp.mode) {
                case kExact: weigh_share(ModeTag<kExact>{}); break;
                case kPot: weigh_share(ModeTag<kPot>{}); break;
                case kPotDrop: weigh_share(ModeTag<kPotDrop>{}); break;
                case kH15: weigh_share(ModeTag<kH15>{}); break;
                default:
                    if constexpr (!HALF) {
                        if (rp.mode == kH15K2) weigh_share(ModeTag<kH15K2>{});
                        else weigh_share(ModeTag<kH15K3>{});
                    }
                    break;
            }
            if (n > 0) add_product(n - 1);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_round);
        }
        // This CTA's part of the result, scaled to the final anchor, into shared memory for the cluster.
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k) {
            const int r = warp + 4 * k;
            if (r < R && lane == 0) {
                fac[r] = ex2_approx((own[k] - (carry[k] == -INFINITY ? 0.f : carry[k])) * p.c);
                mfin[r] = carry[k];
            }
        }
        if constexpr (N == 16) {
#pragma unroll
            for (int r0 = 0; r0 < N; r0 += G) {
                if (r0 < R) {
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1)
#pragma unroll
                        for (int r = r0; r < r0 + G; ++r) l[r] += __shfl_xor_sync(0xffffffffu, l[r], d);
#pragma unroll
                    for (int r = r0; r < r0 + G; ++r)
                        if (lane == r) lw[warp * N + r] = l[r];
                }
            }
        } else {
            reduce_scatter_rows<N>(l, lane, [](float x, float y) { return x + y; });
#pragma unroll
            for (int q = 0; q < N / 32; ++q) lw[warp * N + lane * (N / 32) + q] = l[q];
        }
        named_barrier<1>(128);
        float* part = reinterpret_cast<float*>(ring);   // float[row][D]: the ring is idle by now
        if (kl < D) {
#pragma unroll
            for (int r0 = 0; r0 < N; r0 += G) {
                if (r0 < R) {
#pragma unroll
                    for (int r = r0; r < r0 + G; ++r) part[r * D + kl] = o[r] * fac[r];
                }
            }
        }
        float* lsum = reinterpret_cast<float*>(fix + W::kLOff);
        if (tid < R) lsum[tid] = fac[tid] * ((lw[tid] + lw[N + tid]) + (lw[2 * N + tid] + lw[3 * N + tid]));
    }
    if (warp >= 4) cluster_wait();
    cluster_arrive();
    cluster_wait();      // all parts are in shared memory
    {
        constexpr float kLn2 = 0.6931471805599453f;
        const bool e4m3 = is_exact_like(rp.mode) || rp.mode == kH15K3;
        const float p_off = FP8 ? (e4m3 ? 8.0f : 15.0f) : 0.0f;
        // after an expired wait anywhere in the cluster nothing is stored
        const float flag = lane < cs ? ld_cluster_f32(mapa(sFix + W::kMiscOff + 4, lane)) : 0.0f;
        const bool alive = __all_sync(0xffffffffu, __float_as_int(flag) == 0);
        for (int e = rank * kRowsThreads + tid; e < R * (D / 2); e += cs * kRowsThreads) {
            const int r = e / (D / 2), d = 2 * (e % (D / 2));
            float2 acc = make_float2(0.f, 0.f);
            float lt = 0.f;
#pragma unroll 8
            for (int q = 0; q < cs; ++q) {
                const float2 v = ld_cluster_f32x2(mapa(sRing + (r * D + d) * 4, q));
                lt += ld_cluster_f32(mapa(sFix + W::kLOff + r * 4, q));
                acc.x += v.x;
                acc.y += v.y;
            }
            const float m = mfin[r];
            const bool has_keys = m != -INFINITY && lt > 0.f;
            const float inv = has_keys ? p.v_descale / lt : 0.f;
            const int qi = r / p.group, h = hk * p.group + r % p.group;
            if (alive) {
                const size_t row = (static_cast<size_t>(b) * p.Sq + qi) * p.Hq + h;
                *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(p.o) + row * D + d) = pack_bf16_rn(acc.x * inv, acc.y * inv);
                if (d == 0 && p.lse != nullptr)
                    p.lse[(static_cast<size_t>(b) * p.Hq + h) * p.Sq + qi] = has_keys ? kLn2 * (m * p.c + log2f(lt) - p_off) : -INFINITY;
            }
        }
    }
    cluster_arrive();
    cluster_wait();      // nobody reads this CTA's shared memory any more
    tc_fence_before();
    __syncthreads();
    if (warp == 5) tmem_dealloc(tmem, kRowsCols<N>);
}

// ------------------------------------------------------------------------------------------------
// Host launcher
// ------------------------------------------------------------------------------------------------
namespace {

template <int D, int IN, int N>
struct RowsLauncher {
    static constexpr bool FP8 = IN == kInFP8;
    using W = RowsCfg<D, FP8, N>;
    static constexpr int kTile = TileCfg<D, FP8>::kTileBytes;
    static constexpr int kSmem = kRowsCols<N> == 512 ? 232448 : 115712;    // one or two CTAs per SM (1 KB of each is the system's)
    static constexpr int kSlots = (kSmem - W::kFixedBytes) / kTile < kMaxSlots ? (kSmem - W::kFixedBytes) / kTile : kMaxSlots;
    static_assert(kSlots >= 2 && kSlots * kTile >= N * D * 4, "the ring holds two tiles and the partial result");
    static constexpr int kDynamic = W::kFixedBytes + kSlots * kTile;

    // attr: room for two.  The second one is programmatic dependent launch: the set-up of this kernel overlaps the end of the
    // kernel before it in the stream.
    static void set_cluster(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cs) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cs;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        cfg.blockDim = dim3(kRowsThreads);
        cfg.dynamicSmemBytes = kDynamic;
    }
    // Clusters of `cs` CTAs that the occupancy query says fit the device at once (asked once per device and size).
    static int fit(int dev, int cs) {
        static int known[64][kMaxCluster + 1] = {};
        static bool configured[64] = {};
        auto kern = attn_rows_kernel<D, IN, N>;
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynamic) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
                cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                return 0;
            configured[dev] = true;
        }
        if (known[dev][cs] == 0) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[2];
            set_cluster(cfg, attr, cs);
            cfg.numAttrs = 1;
            cfg.gridDim = dim3(cs);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            known[dev][cs] = n > 0 ? n : -1;
        }
        return known[dev][cs] > 0 ? known[dev][cs] : 0;
    }
    static int plan(const AttnParams& p) {
        int dev = 0, sms = 0;
        if (device_and_sms(&dev, &sms) != cudaSuccess) return 0;
        const RowsShape s{static_cast<double>(p.B) * p.Hkv, (p.Sk + kTileN - 1) / kTileN, N, kTile, static_cast<double>(p.B) * p.Hq, p.Sq * p.group, D};
        const int cs = rows_cluster_size(s, sms, [&](int c) { return fit(dev, c); });
        if (cs == 0 || static_cast<long long>(p.B) * p.Hkv * cs > 0x7fffffffLL) return 0;
        return rows_pay(s, cs, sms) ? cs : 0;
    }
    static cudaError_t launch(int mode, int cs, const CUtensorMap& tk, const CUtensorMap& tv, const void* q, const AttnParams& p,
                              cudaStream_t stream) {
        const long long groups = static_cast<long long>(p.B) * p.Hkv;
        RowsParams rp;
        rp.cs = cs;
        rp.nt = (p.Sk + kTileN - 1) / kTileN;
        constexpr int cap = kRowsCols<N> / N;            // key tiles whose scores fit TMEM
        const int per_cta = (rp.nt + cs - 1) / cs;
        rp.rounds = (per_cta + cap - 1) / cap;
        rp.share = (rp.nt + cs * rp.rounds - 1) / (cs * rp.rounds);
        rp.slots = kSlots;
        rp.rows = p.Sq * p.group;
        rp.mode = mode;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        set_cluster(cfg, attr, cs);
        cfg.gridDim = dim3(static_cast<unsigned>(groups * cs));
        cfg.stream = stream;
        return cudaLaunchKernelEx(&cfg, attn_rows_kernel<D, IN, N>, tk, tv, q, p, rp);
    }
};

// Calls f with the launcher of a combination.
template <int D, int IN, typename F>
void with_rows(int rows, F f) {
    if (rows <= 16) f(RowsLauncher<D, IN, 16>{});
    else if (rows <= 32) f(RowsLauncher<D, IN, 32>{});
    else f(RowsLauncher<D, IN, 64>{});
}
template <typename F>
void with_rows_launcher(int D, int in_type, int rows, F f) {
    if (D == 128) {
        if (in_type == kInBF16) with_rows<128, kInBF16>(rows, f);
        else if (in_type == kInFP16) with_rows<128, kInFP16>(rows, f);
        else with_rows<128, kInFP8>(rows, f);
    } else {
        if (in_type == kInBF16) with_rows<64, kInBF16>(rows, f);
        else if (in_type == kInFP16) with_rows<64, kInFP16>(rows, f);
        else with_rows<64, kInFP8>(rows, f);
    }
}

}  // namespace

// CTAs per (batch, key/value head) for a forward that goes to attn_rows_kernel, 0 for one that does not: it has too many rows,
// a mode the kernel is not built for, no cluster fits the device, or the general path is the faster one (plan.h).
int plan_attn_rows(int D, int in_type, int mode, const AttnParams& p) {
    if (exact_poly_eighths(mode) > 0 || p.tau > 0.0f || static_cast<long long>(p.Sq) * p.group > 64) return 0;
    int cs = 0;
    with_rows_launcher(D, in_type, p.Sq * p.group, [&](auto l) { cs = decltype(l)::plan(p); });
    return cs;
}

cudaError_t launch_attn_rows(int D, int in_type, int mode, int cs, const CUtensorMap& tk, const CUtensorMap& tv, const void* q,
                             const AttnParams& p, cudaStream_t stream) {
    cudaError_t e = cudaErrorInvalidValue;
    with_rows_launcher(D, in_type, p.Sq * p.group, [&](auto l) { e = decltype(l)::launch(mode, cs, tk, tv, q, p, stream); });
    return e;
}

}  // namespace rowmax
