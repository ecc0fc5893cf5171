// Launcher of the split form of the attention forward (attn_fwd_kernel.cuh): a cluster of CTAs shares each work item.
#include "attn_fwd_kernel.cuh"

namespace rowmax {

namespace {

template <int D, int IN, int MODE>
struct SplitLauncher {
    using W = WsCfg<D, IN == kInFP8, true>;

    static void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int parts) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = parts;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        // No programmatic dependent launch, as a precaution: its gain is small if any (512 queries on 16K, bf16 h15, stream of 300
        // calls: 161.9 us with it and 159.9 without in one call; 166.5 without on another machine, where graph replays were
        // 3 % slower too).
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cfg.blockDim = dim3(512);
        cfg.dynamicSmemBytes = W::kSmemBytes;
    }
    // Clusters that fit the device at once (asked once per device and size; 0: none).
    static int fit(int dev, int parts) {
        static int known[64][kMaxSplit + 1] = {};
        if (known[dev][parts] == 0) {
            auto kern = attn_fwd_ws_kernel<D, IN, MODE, true>;
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[1];
            configure(cfg, attr, parts);
            cfg.gridDim = dim3(parts);
            int n = 0;
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, W::kSmemBytes) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            known[dev][parts] = n > 0 ? n : -1;
        }
        return known[dev][parts] > 0 ? known[dev][parts] : 0;
    }
    // CTAs per item (plan.h), 1 for the plain form.
    static int plan(const AttnParams& p, double* steps) {
        int dev = 0, sms = 0;
        if (device_and_sms(&dev, &sms) != cudaSuccess) return 1;
        const int pairs = (p.Sq + 2 * kTileM - 1) / (2 * kTileM);
        const int all = (p.Sk + kTileN - 1) / kTileN;
        const int first_end = p.causal ? 2 * kTileM + p.Sk - p.Sq : p.Sk;
        const int first = first_end <= 0 ? 0 : ((first_end < p.Sk ? first_end : p.Sk) + kTileN - 1) / kTileN;
        const SplitShape s{static_cast<double>(pairs) * p.Hq * p.B, all, first, split_takes_maxima(MODE, IN == kInFP8)};
        return split_parts(s, sms, [&](int parts) { return fit(dev, parts); }, steps);
    }
    static cudaError_t launch(int parts, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, AttnParams p,
                              cudaStream_t stream) {
        const long long items = static_cast<long long>((p.Sq + 2 * kTileM - 1) / (2 * kTileM)) * p.Hq * p.B;
        if (items * parts > 0x7fffffffLL) return cudaErrorInvalidValue;
        p.split = parts;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        configure(cfg, attr, parts);
        cfg.gridDim = dim3(static_cast<unsigned>(items * parts));     // one item per cluster, heaviest first
        cfg.stream = stream;
        return cudaLaunchKernelEx(&cfg, attn_fwd_ws_kernel<D, IN, MODE, true>, tq, tk, tv, p);
    }
};

// Calls f with the launcher of a combination; false for one that has no split form.
template <int D, int IN, typename F>
bool with_mode(int mode, F f) {
    switch (mode) {
        case kExact: f(SplitLauncher<D, IN, kExact>{}); return true;
        case kPot: f(SplitLauncher<D, IN, kPot>{}); return true;
        case kPotDrop: f(SplitLauncher<D, IN, kPotDrop>{}); return true;
        case kH15: f(SplitLauncher<D, IN, kH15>{}); return true;
        default: break;
    }
    if constexpr (IN != kInFP16) {
        switch (mode) {
            case kH15K2: f(SplitLauncher<D, IN, kH15K2>{}); return true;
            case kH15K3: f(SplitLauncher<D, IN, kH15K3>{}); return true;
            default: break;
        }
    }
    return false;
}
template <typename F>
bool with_launcher(int D, int in_type, int mode, F f) {
    if (D == 128) {
        if (in_type == kInBF16) return with_mode<128, kInBF16>(mode, f);
        if (in_type == kInFP16) return with_mode<128, kInFP16>(mode, f);
        return with_mode<128, kInFP8>(mode, f);
    }
    if (in_type == kInBF16) return with_mode<64, kInBF16>(mode, f);
    if (in_type == kInFP16) return with_mode<64, kInFP16>(mode, f);
    return with_mode<64, kInFP8>(mode, f);
}

}  // namespace

// CTAs that should share a work item (1: the plain form), and the estimated time.  A deferred rescale stays whole: its anchor depends on the order.
int plan_attn_split(int D, int in_type, int mode, const AttnParams& p, double* steps) {
    int parts = 1;
    if (!(p.tau > 0.0f)) with_launcher(D, in_type, mode, [&](auto l) { parts = decltype(l)::plan(p, steps); });
    return parts;
}

cudaError_t launch_attn_fwd_split(int D, int in_type, int mode, int parts, const CUtensorMap& tq, const CUtensorMap& tk,
                                  const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
    cudaError_t e = cudaErrorInvalidValue;
    with_launcher(D, in_type, mode, [&](auto l) { e = decltype(l)::launch(parts, tq, tk, tv, p, stream); });
    return e;
}

}  // namespace rowmax
