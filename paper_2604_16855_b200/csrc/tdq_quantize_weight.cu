// tdq_quantize_weight: static per-output-channel symmetric 4-bit weight quantizer (Eq. 4).
// absmax over the row, s_o = max(absmax / 7, 1e-8), then Q = clip(rint(W / s_o), -8, 7), two codes per byte.
//
// Bound by HBM (4 or 2 bytes in, 0.5 out per weight).  weight_rows_kernel reads a row once: one warp (rows of up to 1024
// channels) or a block of up to eight warps keeps it in registers between the maximum and the quantization, with up to
// 32 channels a thread so that all its loads are in flight together, and quantizes two channels at a time with the
// activation quantizer's exact quotient.  Measured, 4096 x 4096: fp32 13.8 us = 5.5 TB/s (a block per row that read it twice and
// divided: 23.5 us), bf16 9.8 us (20.6 us).  weight_quant_kernel keeps what that one does not take: rows of more than
// 8192 channels and padded row lengths that are not a multiple of 8.
#include "tdq_act_group.cuh"
#include "tdq_common.cuh"

namespace tdq {
namespace {

constexpr int kWThreads = 256;

template <bool BF16>
__global__ void __launch_bounds__(kWThreads) weight_quant_kernel(const void* w, int64_t I, int64_t I_pad,
                                                                  uint8_t* wcodes, float* wscale) {
    __shared__ uint32_t warp_max[kWThreads / 32];
    __shared__ float s_shared;
    const int64_t o = blockIdx.x;
    const int64_t base = o * I;
    uint32_t kmax = 0;   // bit pattern of the largest |w|
    for (int64_t i = threadIdx.x; i < I; i += kWThreads) {
        float v = BF16 ? bf16_bits_to_float(reinterpret_cast<const uint16_t*>(w)[base + i])
                       : reinterpret_cast<const float*>(w)[base + i];
        kmax = max(kmax, __float_as_uint(fabsf(v)));
    }
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = kmax;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t m = 0;
        for (int i = 0; i < kWThreads / 32; ++i) m = max(m, warp_max[i]);
        float s = fmaxf(__fdiv_rn(__uint_as_float(m), kQmax), kStepFloor);
        s_shared = s;
        wscale[o] = s;
    }
    __syncthreads();
    const float s = s_shared;
    for (int64_t j = threadIdx.x; j < I_pad / 2; j += kWThreads) {
        int q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int64_t i = 2 * j + h;
            float v = 0.0f;
            if (i < I)
                v = BF16 ? bf16_bits_to_float(reinterpret_cast<const uint16_t*>(w)[base + i])
                         : reinterpret_cast<const float*>(w)[base + i];
            int qi = __float2int_rn(__fdiv_rn(v, s));
            q[h] = max(-8, min(7, qi));
        }
        wcodes[o * (I_pad / 2) + j] = (uint8_t)((q[0] & 0xF) | ((q[1] & 0xF) << 4));
    }
}

// W warps hold a row of at most 256 * NC * W channels; W == 1: four rows per block.
template <bool BF16, int NC, int W>
__global__ void __launch_bounds__(W > 1 ? W * 32 : 128) weight_rows_kernel(const void* w, int64_t O, int32_t I, int32_t I_pad, int32_t load_mode,
                                                                        uint32_t* wcodes, float* wscale) {
    constexpr int kW = BF16 ? 4 : 8;
    __shared__ uint32_t part[W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t o = W > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * 4 + warp;
    if (o >= O) return;
    const int t = W > 1 ? (int)threadIdx.x : lane;
    const uint8_t* src = reinterpret_cast<const uint8_t*>(w) + o * I * (BF16 ? 2 : 4);
    uint32_t x[NC * kW];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int e = (t + c * W * 32) * 8;
#pragma unroll
        for (int j = 0; j < kW; ++j) x[c * kW + j] = 0u;
        if (e + 8 <= I && load_mode == 0) {
#pragma unroll
            for (int h = 0; h < kW / 4; ++h) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + e * (BF16 ? 2 : 4)) + h);
                x[c * kW + 4 * h] = v.x; x[c * kW + 4 * h + 1] = v.y; x[c * kW + 4 * h + 2] = v.z; x[c * kW + 4 * h + 3] = v.w;
            }
        } else if (e < I) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (e + j < I) {
                    if (BF16) x[c * kW + j / 2] |= (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(src) + e + j) << (16 * (j & 1));
                    else x[c * kW + j] = __ldg(reinterpret_cast<const uint32_t*>(src) + e + j);
                }
            }
        }
    }
    uint32_t kmax = 0u;
#pragma unroll
    for (int j = 0; j < NC * kW; ++j) kmax = BF16 ? __vmaxu2(kmax, x[j] & 0x7fff7fffu) : max(kmax, x[j] & 0x7fffffffu);
    if (BF16) kmax = max(kmax & 0xffffu, kmax >> 16) << 16;
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if constexpr (W > 1) {
        if (lane == 0) part[warp] = kmax;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < W; ++i) kmax = max(kmax, part[i]);
    }
    const float s = fmaxf(__fdiv_rn(__uint_as_float(kmax), kQmax), kStepFloor);
    if (t == 0) wscale[o] = s;
    const bool fast = s <= 1e30f;                     // otherwise 1 / s would be subnormal: take the IEEE division
    const float rcp = fast ? __frcp_rn(s) : 0.0f;
    const uint64_t rcp2 = f2_pack(rcp, rcp), neg_s2 = f2_pack(-s, -s), magic2 = f2_pack(kRoundMagic8, kRoundMagic8);
    uint32_t* dst = wcodes + o * (I_pad / 8);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int n = t + c * W * 32;
        if (n * 8 >= I_pad) continue;
        auto get = [&](int j) -> float {
            if (BF16) return (j & 1) ? __uint_as_float(x[c * kW + j / 2] & 0xffff0000u) : __uint_as_float(x[c * kW + j / 2] << 16);
            return __uint_as_float(x[c * kW + (BF16 ? 0 : j)]);
        };
        uint32_t acc = 0u;
        if (fast) {
#pragma unroll
            for (int j = 6; j >= 0; j -= 2) nibbles_fast2(f2_pack(get(j), get(j + 1)), neg_s2, rcp2, magic2, acc);
            acc = pack_word(acc);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) acc |= ((uint32_t)max(-8, min(7, __float2int_rn(__fdiv_rn(get(j), s)))) & 0xFu) << (4 * j);
        }
        dst[n] = acc;
    }
}

template <bool BF16, int NC, int W>
void launch_rows(const void* w, int64_t O, int32_t I, int32_t I_pad, uint8_t* wcodes, float* wscale, cudaStream_t st) {
    const int64_t pitch = (int64_t)I * (BF16 ? 2 : 4);
    const int32_t load_mode = reinterpret_cast<uintptr_t>(w) % 16 == 0 && pitch % 16 == 0 ? 0 : 1;
    const int64_t blocks = W > 1 ? O : (O + 3) / 4;
    weight_rows_kernel<BF16, NC, W><<<(unsigned)blocks, W > 1 ? W * 32 : 128, 0, st>>>(w, O, I, I_pad, load_mode, reinterpret_cast<uint32_t*>(wcodes), wscale);
}
template <bool BF16>
void pick_rows(const void* w, int64_t O, int32_t I, int32_t I_pad, uint8_t* wcodes, float* wscale, cudaStream_t st) {
    if (I_pad <= 256) launch_rows<BF16, 1, 1>(w, O, I, I_pad, wcodes, wscale, st);
    else if (I_pad <= 512) launch_rows<BF16, 2, 1>(w, O, I, I_pad, wcodes, wscale, st);
    else if (I_pad <= 1024) launch_rows<BF16, 4, 1>(w, O, I, I_pad, wcodes, wscale, st);
    else if (I_pad <= 2048) launch_rows<BF16, 4, 2>(w, O, I, I_pad, wcodes, wscale, st);
    else if (I_pad <= 4096) launch_rows<BF16, 4, 4>(w, O, I, I_pad, wcodes, wscale, st);
    else launch_rows<BF16, 4, 8>(w, O, I, I_pad, wcodes, wscale, st);
}

// The affine output correction folded into the layer's constants: a (s Sigma + bias) + b = (a s) Sigma + (a bias + b).
__global__ void fold_affine_kernel(const float* wscale, const float* bias, const float* mul, const float* add, int64_t O,
                                   float* wscale_out, float* bias_out) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= O) return;
    const float a = mul[o];
    wscale_out[o] = __fmul_rn(a, wscale[o]);
    const float ab = bias ? __fmul_rn(a, bias[o]) : 0.0f;
    bias_out[o] = add ? __fadd_rn(ab, add[o]) : ab;
}

}  // namespace
}  // namespace tdq

using namespace tdq;

extern "C" tdq_status tdq_quantize_weight(const void* w, tdq_dtype w_dtype, int64_t O, int64_t I, int32_t pad_to,
                                          uint8_t* wcodes, float* wscale, void* cuda_stream) {
    if (!w || !wcodes || !wscale) return TDQ_ERR_INVALID_ARG;
    if (w_dtype != TDQ_F32 && w_dtype != TDQ_BF16) return TDQ_ERR_INVALID_ARG;
    if (O < 0 || I <= 0 || pad_to < 2 || (pad_to & 1) || O > INT32_MAX) return TDQ_ERR_INVALID_ARG;
    if (O == 0) return TDQ_OK;
    const int64_t I_pad = (I + pad_to - 1) / pad_to * pad_to;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    if (I_pad % 8 == 0 && I_pad <= 8192 && reinterpret_cast<uintptr_t>(wcodes) % 4 == 0) {
        if (w_dtype == TDQ_BF16) pick_rows<true>(w, O, (int32_t)I, (int32_t)I_pad, wcodes, wscale, stream);
        else pick_rows<false>(w, O, (int32_t)I, (int32_t)I_pad, wcodes, wscale, stream);
    } else if (w_dtype == TDQ_BF16)
        weight_quant_kernel<true><<<(unsigned)O, kWThreads, 0, stream>>>(w, I, I_pad, wcodes, wscale);
    else
        weight_quant_kernel<false><<<(unsigned)O, kWThreads, 0, stream>>>(w, I, I_pad, wcodes, wscale);
    if (cudaGetLastError() != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

extern "C" tdq_status tdq_fold_output_affine(const float* wscale, const float* bias, const float* out_mul, const float* out_add,
                                             int64_t O, float* wscale_out, float* bias_out, void* cuda_stream) {
    if (!wscale || !out_mul || !wscale_out || !bias_out) return TDQ_ERR_INVALID_ARG;
    if (O < 0 || O > INT32_MAX) return TDQ_ERR_INVALID_ARG;
    if (O == 0) return TDQ_OK;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    fold_affine_kernel<<<(unsigned)((O + 255) / 256), 256, 0, stream>>>(wscale, bias, out_mul, out_add, O, wscale_out, bias_out);
    if (cudaGetLastError() != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}
