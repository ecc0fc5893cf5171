// Launcher of the two-stream form of the attention forward (attn_streams_kernel.cuh).
#include "attn_streams_kernel.cuh"

namespace rowmax {

namespace {

template <int D, int IN, int MODE, bool PAIR>
struct StreamsLauncher {
    using W = StreamsCfg<D, IN == kInFP8, PAIR>;
    static constexpr int kCtas = PAIR ? 2 : 1;

    static void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
        // Programmatic dependent launch as in the plain form; used where every CTA has one item.
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = kCtas;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.blockDim = dim3(512);
        cfg.dynamicSmemBytes = W::kSmemBytes;
    }
    // CTAs, or pairs of them, that fit the device at once (asked once per device; 0: none).
    static int fit() {
        static int known[64] = {};
        int dev = 0, sms = 0;
        if (device_and_sms(&dev, &sms) != cudaSuccess) return 0;
        if (known[dev] == 0) {
            auto kern = attn_fwd_streams_kernel<D, IN, MODE, PAIR>;
            int n = sms;
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, W::kSmemBytes);
            if (PAIR && e == cudaSuccess) {
                cudaLaunchConfig_t cfg = {};
                cudaLaunchAttribute attr[2];
                configure(cfg, attr);
                cfg.attrs = attr + 1;
                cfg.numAttrs = 1;
                cfg.gridDim = dim3(kCtas);
                e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
            }
            if (e != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            known[dev] = n > 0 ? n : -1;
        }
        return known[dev] > 0 ? known[dev] : 0;
    }
    static cudaError_t launch(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
        const int places = fit();
        const long long items = static_cast<long long>((p.Sq + kCtas * kTileM - 1) / (kCtas * kTileM)) * p.Hq * p.B;
        if (places == 0 || items > 0x3fffffffLL) return cudaErrorInvalidValue;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        configure(cfg, attr);
        cfg.gridDim = dim3(kCtas * static_cast<unsigned>(items < places ? items : places));
        cfg.stream = stream;
        const bool early = items <= places;
        cfg.attrs = early ? attr : attr + 1;
        cfg.numAttrs = (early ? 1 : 0) + (PAIR ? 1 : 0);
        return cudaLaunchKernelEx(&cfg, attn_fwd_streams_kernel<D, IN, MODE, PAIR>, tq, tk, tv, p);
    }
};

// Calls f with the launcher of a combination; false for one that has no two-stream form.
template <int D, int IN, bool PAIR, typename F>
bool with_mode(int mode, F f) {
    switch (mode) {
        case kExact: f(StreamsLauncher<D, IN, kExact, PAIR>{}); return true;
        case kPot: f(StreamsLauncher<D, IN, kPot, PAIR>{}); return true;
        case kPotDrop: f(StreamsLauncher<D, IN, kPotDrop, PAIR>{}); return true;
        case kH15: f(StreamsLauncher<D, IN, kH15, PAIR>{}); return true;
        default: break;
    }
    if constexpr (IN != kInFP16) {
        switch (mode) {
            case kH15K2: f(StreamsLauncher<D, IN, kH15K2, PAIR>{}); return true;
            case kH15K3: f(StreamsLauncher<D, IN, kH15K3, PAIR>{}); return true;
            default: break;
        }
    }
    return false;
}
template <typename F>
bool with_launcher(int D, int in_type, int mode, bool pair, F f) {
    if (D == 128 && pair) {
        if (in_type == kInBF16) return with_mode<128, kInBF16, true>(mode, f);
        if (in_type == kInFP16) return with_mode<128, kInFP16, true>(mode, f);
        return with_mode<128, kInFP8, true>(mode, f);
    }
    if (D == 128) {
        if (in_type == kInBF16) return with_mode<128, kInBF16, false>(mode, f);
        if (in_type == kInFP16) return with_mode<128, kInFP16, false>(mode, f);
        return with_mode<128, kInFP8, false>(mode, f);
    }
    if (pair) return false;
    if (in_type == kInBF16) return with_mode<64, kInBF16, false>(mode, f);
    if (in_type == kInFP16) return with_mode<64, kInFP16, false>(mode, f);
    return with_mode<64, kInFP8, false>(mode, f);
}

}  // namespace

cudaError_t launch_attn_fwd_streams(int D, int in_type, int mode, bool pair, const CUtensorMap& tq, const CUtensorMap& tk,
                                    const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
    cudaError_t e = cudaErrorInvalidValue;
    with_launcher(D, in_type, mode, pair, [&](auto l) { e = decltype(l)::launch(tq, tk, tv, p, stream); });
    return e;
}

}  // namespace rowmax
