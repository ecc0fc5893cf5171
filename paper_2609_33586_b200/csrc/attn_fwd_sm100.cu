// Launcher of the attention forward (attn_fwd_kernel.cuh) and the weight-map kernels.
#include "attn_fwd_kernel.cuh"

namespace rowmax {

// ------------------------------------------------------------------------------------------------
// Host launcher
// ------------------------------------------------------------------------------------------------
template <int D, int IN>
static cudaError_t dispatch_mode(int mode, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                 const AttnParams& p, cudaStream_t stream) {
    switch (mode) {
        case kExact: return launch_ws<D, IN, kExact>(tq, tk, tv, p, stream);
        case kPot: return launch_ws<D, IN, kPot>(tq, tk, tv, p, stream);
        case kPotDrop: return launch_ws<D, IN, kPotDrop>(tq, tk, tv, p, stream);
        case kH15: return launch_ws<D, IN, kH15>(tq, tk, tv, p, stream);
        default: break;
    }
    if constexpr (IN != kInFP16) {   // the family members and the emulated control are built for bf16 and fp8 only
        switch (mode) {
            case kH15K2: return launch_ws<D, IN, kH15K2>(tq, tk, tv, p, stream);
            case kH15K3: return launch_ws<D, IN, kH15K3>(tq, tk, tv, p, stream);
            case kExactPoly: return launch_ws<D, IN, kExactPoly>(tq, tk, tv, p, stream);
            default: break;
        }
        if constexpr (D == 128) {   // the other emulation shares: the paper's main head dimension only
            switch (mode) {
                case kExactPoly1: return launch_ws<D, IN, kExactPoly1>(tq, tk, tv, p, stream);
                case kExactPoly3: return launch_ws<D, IN, kExactPoly3>(tq, tk, tv, p, stream);
                case kExactPoly4: return launch_ws<D, IN, kExactPoly4>(tq, tk, tv, p, stream);
                default: break;
            }
        }
    }
    return cudaErrorInvalidValue;
}

// Returns cudaErrorInvalidValue for a combination that is not built.
cudaError_t launch_attn_fwd(int D, int in_type, int mode, const CUtensorMap& tq, const CUtensorMap& tk,
                            const CUtensorMap& tv, const AttnParams& p, cudaStream_t stream) {
    if (in_type == kInBF16 && D == 128) return dispatch_mode<128, kInBF16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInBF16 && D == 64) return dispatch_mode<64, kInBF16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP16 && D == 128) return dispatch_mode<128, kInFP16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP16 && D == 64) return dispatch_mode<64, kInFP16>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP8 && D == 128) return dispatch_mode<128, kInFP8>(mode, tq, tk, tv, p, stream);
    if (in_type == kInFP8 && D == 64) return dispatch_mode<64, kInFP8>(mode, tq, tk, tv, p, stream);
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------------------------------------
// Weight-map sweep: the same device functions on a flat array of offsets.
// ------------------------------------------------------------------------------------------------
__global__ void weight_map_kernel(const float* __restrict__ x, float* __restrict__ w, size_t n, int mode,
                                  uint32_t two22) {
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float xi = x[i];
        float wi;
        if (mode == kExact) wi = w_exact(xi);
        else if (mode == kExactPoly) wi = w_exact_poly3(xi);
        else if (mode == kPot) wi = w_pot(xi);
        else {
            // both lanes of the pair function are exercised: even indices take the shift-add lane, odd
            // indices the multiply-add lane
            float2 r;
            if (mode == kH15K2) r = w_h15_doubled_pair<0, true, 2>(make_float2(xi * 4.0f, xi * 4.0f), two22);
            else if (mode == kH15K3) r = w_h15_doubled_pair<0, true, 3>(make_float2(xi * 8.0f, xi * 8.0f), two22);
            else r = w_h15_doubled_pair<0, true, 1>(make_float2(xi * 2.0f, xi * 2.0f), two22);
            wi = (i & 1) ? r.y : r.x;
        }
        w[i] = wi;
    }
}

// Rowmax-PoT with a run-time tail (index cap K_max, clamped or dropped), the function of the 16-bit paths.
__global__ void weight_map_pot_kernel(const float* __restrict__ x, float* __restrict__ w, size_t n, int kmax, int drop) {
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride)
        w[i] = w_pot_tail(x[i], kmax, drop != 0);
}

cudaError_t launch_weight_map_pot(const float* x, float* w, size_t n, int kmax, int drop, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    size_t blocks = (n + 255) / 256;
    if (blocks > 148 * 8) blocks = 148 * 8;
    weight_map_pot_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(x, w, n, kmax, drop);
    return cudaGetLastError();
}

// The weights as the fused kernel's hot loop produces and stores them: every thread takes 32 consecutive offsets
// as one chunk of a score row (score = offset, scale 1, anchor 0), runs weights_chunk32 with the template
// arguments of the fused kernel for that storage type (fp8: its choice between the unclamped and the clamped h15
// variant, here per chunk, in the fused kernel per warp and key tile; 16 bit: the saturating form), and decodes
// the packed P words back to fp32, divided by the P scale.
template <bool FP8, bool HALF, int MODE>
__global__ void weight_map_fused_kernel(const float* __restrict__ x, float* __restrict__ w, size_t n, uint32_t two22,
                                        float pot_neg_cap, float pot_drop_x) {
    constexpr int kFam = h15_family_k(MODE);
    constexpr int kOff = PFormat<FP8, MODE>::kOffLog2;
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t chunk = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; chunk * 32 < n; chunk += stride) {
        uint32_t s[32];
        float lowest = INFINITY;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const size_t idx = chunk * 32 + i;
            const float xi = idx < n ? x[idx] : 0.0f;
            s[i] = __float_as_uint(xi);
            lowest = fminf(lowest, xi);
        }
        RowScale rs;
        const float c_row = static_cast<float>(1 << kFam);
        const float nmc = is_exact_like(MODE) ? static_cast<float>(kOff) : 0.0f;
        rs.c = make_float2(c_row, c_row);
        rs.nmc = make_float2(nmc, nmc);
        rs.two22 = two22;
        rs.pot_neg_cap = pot_neg_cap;
        rs.pot_drop_x = pot_drop_x;
        rs.clamp_lo = 0.f;
        if constexpr (kFam > 0) rs.clamp_lo = h15_clamp_floor<kFam>();
        float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        uint32_t pw[16];
        if constexpr (kFam > 0 && !FP8) {
            // 16-bit inputs: the saturating form, as in a key tile without masked scores
            constexpr float kR = 126.0f * (1 << kFam);
            rs.su = -static_cast<float>(1 << kFam) * (1.0f / kR);
            rs.ou = make_float2(0.0f, 0.0f);
            rs.sat_mul = -kR;
            weights_chunk32<FP8, MODE, false, true, HALF, true>(s, rs, 32, acc, pw);
        } else {
            const bool clamp = kFam > 0 && !(lowest * (1 << kFam) >= -125.0f * (1 << kFam));
            if (clamp) weights_chunk32<FP8, MODE, false, true, HALF>(s, rs, 32, acc, pw);
            else weights_chunk32<FP8, MODE, false, false, HALF>(s, rs, 32, acc, pw);
        }
        const float unscale = __uint_as_float(static_cast<uint32_t>(127 - kOff) << 23);   // 2^-kOff
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float v;
            if constexpr (FP8) {
                const uint32_t byte = (pw[i / 4] >> (8 * (i % 4))) & 0xFFu;
                if constexpr (PFormat<FP8, MODE>::kE4M3) {
                    uint32_t h2;
                    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(static_cast<uint16_t>(byte)));
                    v = __half2float(__ushort_as_half(static_cast<unsigned short>(h2 & 0xFFFFu)));
                } else {
                    v = __half2float(__ushort_as_half(static_cast<unsigned short>(byte << 8)));   // e5m2 = upper byte of fp16
                }
            } else {
                const uint32_t h = (pw[i / 2] >> (16 * (i % 2))) & 0xFFFFu;
                if constexpr (HALF) v = __half2float(__ushort_as_half(static_cast<unsigned short>(h)));
                else v = __uint_as_float(h << 16);
            }
            const size_t idx = chunk * 32 + i;
            if (idx < n) w[idx] = v * unscale;
        }
    }
}

template <bool FP8, bool HALF>
static cudaError_t launch_fused_map_mode(const float* x, float* w, size_t n, int mode, float pot_neg_cap, float pot_drop_x,
                                         cudaStream_t stream) {
    size_t blocks = ((n + 31) / 32 + 127) / 128;
    if (blocks > 148 * 8) blocks = 148 * 8;
    const unsigned g = static_cast<unsigned>(blocks);
    switch (mode) {
        case kExact: weight_map_fused_kernel<FP8, HALF, kExact><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
        case kPot: weight_map_fused_kernel<FP8, HALF, kPot><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
        case kPotDrop: weight_map_fused_kernel<FP8, HALF, kPotDrop><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
        case kH15: weight_map_fused_kernel<FP8, HALF, kH15><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
        default:
            if constexpr (!HALF) {
                switch (mode) {
                    case kH15K2: weight_map_fused_kernel<FP8, HALF, kH15K2><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
                    case kH15K3: weight_map_fused_kernel<FP8, HALF, kH15K3><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
                    case kExactPoly: weight_map_fused_kernel<FP8, HALF, kExactPoly><<<g, 128, 0, stream>>>(x, w, n, 1u << 22, pot_neg_cap, pot_drop_x); break;
                    default: return cudaErrorInvalidValue;
                }
            } else {
                return cudaErrorInvalidValue;
            }
    }
    return cudaGetLastError();
}

cudaError_t launch_weight_map_fused(const float* x, float* w, size_t n, int mode, int in_type, float pot_neg_cap,
                                    float pot_drop_x, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    if (in_type == kInFP8) return launch_fused_map_mode<true, false>(x, w, n, mode, pot_neg_cap, pot_drop_x, stream);
    if (in_type == kInFP16) return launch_fused_map_mode<false, true>(x, w, n, mode, pot_neg_cap, pot_drop_x, stream);
    return launch_fused_map_mode<false, false>(x, w, n, mode, pot_neg_cap, pot_drop_x, stream);
}

cudaError_t launch_weight_map(const float* x, float* w, size_t n, int mode, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    const int threads = 256;
    size_t blocks = (n + threads - 1) / threads;
    if (blocks > 148 * 8) blocks = 148 * 8;
    weight_map_kernel<<<static_cast<unsigned>(blocks), threads, 0, stream>>>(x, w, n, mode, 1u << 22);
    return cudaGetLastError();
}

// One warp waits on a barrier nobody arrives on, with a short limit: the wait gives up, records its code in the
// status word and the kernel returns.  Exercises the bounded-wait path without touching the attention kernels.
__global__ void selftest_wait_kernel(int* status, long long limit_cycles) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int cta_abort;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bar), 1);
        cta_abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    const WaitCtx ctx{smem_u32(&cta_abort), status, limit_cycles};
    mbar_wait(smem_u32(&bar), 0, ctx, (kRoleSelftest << 8) | kBarSelftest);
}

cudaError_t launch_selftest_wait(int* status, long long limit_cycles, cudaStream_t stream) {
    selftest_wait_kernel<<<1, 32, 0, stream>>>(status, limit_cycles);
    return cudaGetLastError();
}

cudaError_t device_and_sms(int* dev, int* sms) {
    static int known[64] = {};
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    if (*dev < 0 || *dev >= 64) return cudaErrorInvalidDevice;
    if (known[*dev] == 0) {
        e = cudaDeviceGetAttribute(&known[*dev], cudaDevAttrMultiProcessorCount, *dev);
        if (e != cudaSuccess) return e;
    }
    *sms = known[*dev];
    return cudaSuccess;
}

__device__ int g_attn_status = 0;

cudaError_t status_word_address(int** out) {
    return cudaGetSymbolAddress(reinterpret_cast<void**>(out), g_attn_status);
}

}  // namespace rowmax
