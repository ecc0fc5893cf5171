// Launcher of the two-stream form of the attention forward (attn_streams_kernel.cuh).
#include "attn_streams_kernel.cuh"

namespace rowmax {

namespace {

template <int D, int IN, int MODE>
cudaError_t launch_streams(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
    using W = StreamsCfg<D, IN == kInFP8>;
    auto kern = attn_fwd_streams_kernel<D, IN, MODE>;
    static bool configured[64] = {};   // per device: the shared-memory opt-in of this instance
    int dev = 0, sm_count = 0;
    cudaError_t e = device_and_sms(&dev, &sm_count);
    if (e != cudaSuccess) return e;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, W::kSmemBytes);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    const long long items = static_cast<long long>((p.Sq + kTileM - 1) / kTileM) * p.Hq * p.B;
    if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr;      // programmatic dependent launch where every CTA has one item, as in the plain form
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(items < sm_count ? items : sm_count));
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = W::kSmemBytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = items <= sm_count ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, tq, tk, tv, p);
}

template <int D, int IN>
cudaError_t dispatch_mode(int mode, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p,
                          cudaStream_t stream) {
    switch (mode) {
        case kExact: return launch_streams<D, IN, kExact>(tq, tk, tv, p, stream);
        case kPot: return launch_streams<D, IN, kPot>(tq, tk, tv, p, stream);
        case kPotDrop: return launch_streams<D, IN, kPotDrop>(tq, tk, tv, p, stream);
        case kH15: return launch_streams<D, IN, kH15>(tq, tk, tv, p, stream);
        default: break;
    }
    if constexpr (IN != kInFP16) {
        switch (mode) {
            case kH15K2: return launch_streams<D, IN, kH15K2>(tq, tk, tv, p, stream);
            case kH15K3: return launch_streams<D, IN, kH15K3>(tq, tk, tv, p, stream);
            default: break;
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Whether a forward takes this form; parts and split_steps: what the split form would make of it (1: the plain form).  The
// emulated controls and a deferred rescale have no instances here.
bool plan_attn_streams(int D, int in_type, int mode, int parts, double split_steps, const AttnParams& p) {
    if (p.tau > 0.0f || exact_poly_eighths(mode) > 0) return false;
    int dev = 0, sms = 0;
    if (device_and_sms(&dev, &sms) != cudaSuccess) return false;
    const StreamShape s{static_cast<long long>(p.Hq) * p.B, p.Sq, p.Sk, D, p.causal != 0, is_exact_like(mode), in_type == kInFP8};
    return streams_pay(s, parts, split_steps, sms);
}

cudaError_t launch_attn_fwd_streams(int D, int in_type, int mode, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                    const AttnParams& p, cudaStream_t stream) {
    if (in_type == kInBF16 && D == 128) return dispatch_mode<128, kInBF16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInBF16 && D == 64) return dispatch_mode<64, kInBF16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP16 && D == 128) return dispatch_mode<128, kInFP16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP16 && D == 64) return dispatch_mode<64, kInFP16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP8 && D == 128) return dispatch_mode<128, kInFP8>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP8 && D == 64) return dispatch_mode<64, kInFP8>(mode, tq, tk, tv, p, stream);
    return cudaErrorInvalidValue;
}

}  // namespace rowmax
