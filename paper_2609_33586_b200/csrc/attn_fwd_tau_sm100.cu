// The deferred-rescale instances of the attention forward (attn_fwd_tau; bf16 inputs).
#include "attn_fwd_kernel.cuh"

namespace rowmax {

template <int D>
static cudaError_t dispatch_tau(int mode, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                const AttnParams& p, cudaStream_t stream) {
    switch (mode) {
        case kExact: return launch_ws<D, kInBF16, kExact, true>(tq, tk, tv, p, stream);
        case kPot: return launch_ws<D, kInBF16, kPot, true>(tq, tk, tv, p, stream);
        case kH15: return launch_ws<D, kInBF16, kH15, true>(tq, tk, tv, p, stream);
        case kH15K2: return launch_ws<D, kInBF16, kH15K2, true>(tq, tk, tv, p, stream);
        case kH15K3: return launch_ws<D, kInBF16, kH15K3, true>(tq, tk, tv, p, stream);
        case kExactPoly: return launch_ws<D, kInBF16, kExactPoly, true>(tq, tk, tv, p, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_attn_fwd_tau(int D, int mode, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                const AttnParams& p, cudaStream_t stream) {
    return D == 128 ? dispatch_tau<128>(mode, tq, tk, tv, p, stream) : dispatch_tau<64>(mode, tq, tk, tv, p, stream);
}

}  // namespace rowmax
