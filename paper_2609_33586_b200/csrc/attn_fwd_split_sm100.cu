// Launcher of the split form of the attention forward (attn_fwd_kernel.cuh): a cluster of CTAs shares each work item.
#include "attn_fwd_kernel.cuh"

#include <cmath>

namespace rowmax {

namespace {

template <int D, int IN, int MODE>
struct SplitLauncher {
    using W = WsCfg<D, IN == kInFP8, true>;

    static void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int parts) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = parts;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see launch_ws
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        cfg.blockDim = dim3(512);
        cfg.dynamicSmemBytes = W::kSmemBytes;
    }
    // Clusters that fit the device at once (asked once per device and size; 0: none).
    static int fit(int dev, int parts) {
        static int known[64][kMaxSplit + 1] = {};
        if (known[dev][parts] == 0) {
            auto kern = attn_fwd_ws_kernel<D, IN, MODE, true>;
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[2];
            configure(cfg, attr, parts);
            cfg.numAttrs = 1;
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
    static cudaError_t launch(int parts, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, AttnParams p,
                              cudaStream_t stream) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        const int n = fit(dev, parts);
        if (n <= 0) return cudaErrorInvalidConfiguration;
        const long long items = static_cast<long long>((p.Sq + 2 * kTileM - 1) / (2 * kTileM)) * p.Hq * p.B;
        p.split = parts;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        configure(cfg, attr, parts);
        if (items * parts > 0x7fffffffLL) return cudaErrorInvalidValue;
        cfg.gridDim = dim3(static_cast<unsigned>(items * parts));     // one item per cluster, heaviest first
        cfg.stream = stream;
        return cudaLaunchKernelEx(&cfg, attn_fwd_ws_kernel<D, IN, MODE, true>, tq, tk, tv, p);
    }
};

template <int D, int IN>
cudaError_t split_mode(int mode, int parts, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                       const AttnParams& p, cudaStream_t stream) {
    switch (mode) {
        case kExact: return SplitLauncher<D, IN, kExact>::launch(parts, tq, tk, tv, p, stream);
        case kPot: return SplitLauncher<D, IN, kPot>::launch(parts, tq, tk, tv, p, stream);
        case kPotDrop: return SplitLauncher<D, IN, kPotDrop>::launch(parts, tq, tk, tv, p, stream);
        case kH15: return SplitLauncher<D, IN, kH15>::launch(parts, tq, tk, tv, p, stream);
        default: break;
    }
    if constexpr (IN != kInFP16) {
        switch (mode) {
            case kH15K2: return SplitLauncher<D, IN, kH15K2>::launch(parts, tq, tk, tv, p, stream);
            case kH15K3: return SplitLauncher<D, IN, kH15K3>::launch(parts, tq, tk, tv, p, stream);
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace

int plan_split(int mode, const AttnParams& p) {
    (void)mode; (void)p;
    return 1;
}

cudaError_t launch_attn_fwd_split(int D, int in_type, int mode, int parts, const CUtensorMap& tq, const CUtensorMap& tk,
                                  const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
    if (D == 128) {
        if (in_type == kInBF16) return split_mode<128, kInBF16>(mode, parts, tq, tk, tv, p, stream);
        if (in_type == kInFP16) return split_mode<128, kInFP16>(mode, parts, tq, tk, tv, p, stream);
        return split_mode<128, kInFP8>(mode, parts, tq, tk, tv, p, stream);
    }
    if (in_type == kInBF16) return split_mode<64, kInBF16>(mode, parts, tq, tk, tv, p, stream);
    if (in_type == kInFP16) return split_mode<64, kInFP16>(mode, parts, tq, tk, tv, p, stream);
    return split_mode<64, kInFP8>(mode, parts, tq, tk, tv, p, stream);
}

}  // namespace rowmax
