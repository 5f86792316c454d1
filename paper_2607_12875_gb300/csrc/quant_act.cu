// Activation rows as two e4m3 codes per value, the operand of the fp8 tensor
// cores: with one power of two s per row and 128 consecutive values, v = x / s
// (exact), q1 = e4m3(v) and q2 = e4m3((v - q1) * 2^kLow), so that x is
// s * (q1 + 2^-kLow * q2). A bf16 value has 8 significant bits and the two codes
// hold 4 each; what limits them is e4m3's lowest bit, 2^-9.
//   kLow = 5 (feature-major GEMM, which scales the second codes' sums apart): s
//     brings the block's largest magnitude into [128, 256), so that q2 just fits;
//     x is exact for every |v| >= 2^-7 and within 2^-15 * s below that, 2^-22 of
//     the block's largest value. What is left over there goes into a second pair
//     of codes, 2^kWideBits further down, if it belongs to more than an eighth of
//     the block's nonzero values: exact to 2^-44 of the largest. The GEMM walks k a
//     second time, with those planes, when any block set the flag. (A block that
//     leaves less has all its inexact values below the others, and they are few:
//     2^-11 of the others' part of a sum at most. Normal rows leave one value in
//     10^4. 16 experts, weights of 0 at one channel 2^16 times the rest: output
//     within 2.9e-3 of 64 bits with the second pair, 1.4e-2 without; bf16 rounding
//     alone gives 2.9e-3.) Blocks without one have zeros there, so that a row's
//     outputs do not depend on other rows.
//   kLow = 0 (row-major fp8 GEMM, which adds both codes' products up in the same
//     columns): s brings it into [224, 448], as far up as e4m3 goes; x is exact
//     for every |v| >= 2^-2 and within 2^-10 * s below that.
//
// Bound by its writes (two codes per value) once there are rows enough. One
// warp takes 4 blocks of a row, not a whole row: 48 rows of 7168 quantised in
// 4.2 us against 22.4 us with a warp per row, and the exact scaling needs no
// division (16384 gathered rows: see launch_quant_scatter).
#include <cuda_fp8.h>

#include "common.cuh"
#include "kernels.h"

namespace gbmoe {

constexpr int QB = 128;   // values per scale
constexpr int QU = 4;     // blocks of a row per warp, their loads in flight together
constexpr int QWARPS = 8;

__device__ __forceinline__ uint32_t e4m3x2(float a, float b) {
    return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
}

// kFourBit: the order that 4-bit weights are decoded in (ffn_fm.cu): within 8
// consecutive values the even ones come before the odd ones.
//
// Rows of src [*, K] -> code planes q [2 or (kLow > 0) 4][n_rows][K] and scales s
// [n_rows][K/128]. Row r reads source row gather[r] / gather_div (r itself
// without gather; a negative entry gives a zero row). With scatter, source row
// r is quantised once and written to the n_copies rows scatter[r * n_copies ..]
// (a negative entry: none); q and s then hold n_rows * n_copies rows. Lane l takes elements
// 4l .. 4l+3 of a block. A block that holds an infinity gets the codes +-1
// there, 0 elsewhere and an infinite scale, so its sums are infinite as they
// should be; a NaN makes the scale NaN.
template <bool kFourBit, bool kScatter, int kLow>
__global__ void __launch_bounds__(QWARPS * 32)
quant_rows_kernel(const __nv_bfloat16* __restrict__ src, const int32_t* __restrict__ gather, int gather_div,
                  const int32_t* __restrict__ scatter, int n_copies,
                  int64_t n_rows, int K, uint8_t* __restrict__ q, float* __restrict__ s, int32_t* __restrict__ wide,
                  const int32_t* __restrict__ kept, int64_t n_routed) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int nblk = K / QB, parts = (nblk + QU - 1) / QU;
    const int64_t plane = n_rows * (kScatter ? n_copies : 1) * K;
    uint8_t* q2 = q + plane;
    const int64_t first_left_out = kept ? *kept : n_routed;
    const int64_t units = n_rows * parts;
    for (int64_t w = (int64_t)blockIdx.x * QWARPS + (threadIdx.x >> 5); w < units; w += (int64_t)gridDim.x * QWARPS) {
        const int64_t r = w / parts;
        const int b0 = (int)(w - r * parts) * QU;
        if (r >= first_left_out && r < n_routed) continue;
        int64_t from = r;
        if (gather) {
            const int32_t g = gather[r];
            from = g >= 0 ? g / gather_div : -1;
        }
        uint2 raw[QU];
#pragma unroll
        for (int u = 0; u < QU; ++u) {
            raw[u] = make_uint2(0, 0);
            if (from >= 0 && b0 + u < nblk)
                raw[u] = *reinterpret_cast<const uint2*>(src + from * K + (b0 + u) * QB + 4 * lane);
        }
#pragma unroll
        for (int u = 0; u < QU; ++u) {
            const int b = b0 + u;
            if (b >= nblk) break;
            const float v[4] = {bf16lo(raw[u].x), bf16hi(raw[u].x), bf16lo(raw[u].y), bf16hi(raw[u].y)};
            // the largest magnitude as float bits: they order like the values, NaN above infinity
            uint32_t m = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) m = max(m, __float_as_uint(v[i]) & 0x7fffffffu);
            m = __reduce_max_sync(0xffffffffu, m);
            // s = 2^(exponent of the largest - 7), or - 8 where it then is at most 448; at least 2^-126
            const int e = max((int)(m >> 23) - (kLow == 0 && (m & 0x7fffffu) <= 0x600000u ? 8 : 7), 1);
            float sc = __uint_as_float((uint32_t)e << 23);
            float t[4];
            if (m < 0x7f800000u) {
                const float inv = __uint_as_float((uint32_t)(254 - e) << 23);  // 1 / s, exact (1 <= e <= 247)
#pragma unroll
                for (int i = 0; i < 4; ++i) t[i] = v[i] * inv;
            } else {
                sc = __uint_as_float(m == 0x7f800000u ? 0x7f800000u : 0x7fc00000u);
#pragma unroll
                for (int i = 0; i < 4; ++i) t[i] = isinf(v[i]) ? copysignf(1.0f, v[i]) : 0.0f;
            }
            const uint32_t a = e4m3x2(t[0], t[1]) | (e4m3x2(t[2], t[3]) << 16);
            const float2 lo = e4m3x2_to_f32x2(a & 0xffffu), hi = e4m3x2_to_f32x2(a >> 16);
            constexpr float kUp = 1 << kLow;
            const float rr[4] = {(t[0] - lo.x) * kUp, (t[1] - lo.y) * kUp, (t[2] - hi.x) * kUp, (t[3] - hi.y) * kUp};
            const uint32_t a2 = e4m3x2(rr[0], rr[1]) | (e4m3x2(rr[2], rr[3]) << 16);
            uint32_t a3 = 0, a4 = 0;
            if constexpr (kLow > 0) {
                const float2 lo2 = e4m3x2_to_f32x2(a2 & 0xffffu), hi2 = e4m3x2_to_f32x2(a2 >> 16);
                float left[4] = {rr[0] - lo2.x, rr[1] - lo2.y, rr[2] - hi2.x, rr[3] - hi2.y};
                int n = 0;  // values that leave something over, and 2^16 times the nonzero ones
#pragma unroll
                for (int i = 0; i < 4; ++i) n += (left[i] != 0.0f) + ((t[i] != 0.0f) << 16);
                n = __reduce_add_sync(0xffffffffu, n);
                if (8 * (n & 0xffff) > n >> 16) {
                    constexpr float kDown = 1 << (kWideBits - kLow);
#pragma unroll
                    for (int i = 0; i < 4; ++i) left[i] *= kDown;
                    a3 = e4m3x2(left[0], left[1]) | (e4m3x2(left[2], left[3]) << 16);
                    const float2 lo3 = e4m3x2_to_f32x2(a3 & 0xffffu), hi3 = e4m3x2_to_f32x2(a3 >> 16);
                    a4 = e4m3x2((left[0] - lo3.x) * kUp, (left[1] - lo3.y) * kUp) |
                         (e4m3x2((left[2] - hi3.x) * kUp, (left[3] - hi3.y) * kUp) << 16);
                    if (lane == 0) *wide = 1;
                }
            }
            if constexpr (kFourBit) {
                // this lane's values are 0..3 (even lane) or 4..7 of 8: the even two, then the odd two
                const int64_t at = r * K + b * QB + 8 * (lane >> 1) + 2 * (lane & 1);
                const uint32_t codes[4] = {a, a2, a3, a4};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    *reinterpret_cast<uint16_t*>(q + i * plane + at) = (uint16_t)__byte_perm(codes[i], 0, 0x4420);
                    *reinterpret_cast<uint16_t*>(q + i * plane + at + 4) = (uint16_t)__byte_perm(codes[i], 0, 0x4431);
                }
            } else {
                auto put = [&](int64_t to) {
                    const int64_t at = to * K + b * QB + 4 * lane;
                    *reinterpret_cast<uint32_t*>(q + at) = a;
                    *reinterpret_cast<uint32_t*>(q2 + at) = a2;
                    if constexpr (kLow > 0) {
                        *reinterpret_cast<uint32_t*>(q2 + plane + at) = a3;
                        *reinterpret_cast<uint32_t*>(q2 + 2 * plane + at) = a4;
                    }
                    if (lane == 0) s[to * nblk + b] = sc;
                };
                if constexpr (kScatter) {
                    for (int c = 0; c < n_copies; ++c)
                        if (const int32_t to = scatter[r * n_copies + c]; to >= 0) put(to);
                } else {
                    put(r);
                }
            }
            if (kFourBit && lane == 0) s[r * nblk + b] = sc;
        }
    }
}

template <bool kFourBit, bool kScatter, int kLow>
static cudaError_t launch_quant(const void* src, const int32_t* gather, int gather_div, const int32_t* scatter,
                                int n_copies, int64_t n_rows, int K, void* q, float* s, int32_t* wide,
                                const int32_t* kept, int64_t n_routed, cudaStream_t stream) {
    const int64_t units = n_rows * ((K / QB + QU - 1) / QU);
    const int blocks = (int)min64((units + QWARPS - 1) / QWARPS, (int64_t)sm_count() * 16);
    if (blocks <= 0) return cudaSuccess;
    return launch_k(quant_rows_kernel<kFourBit, kScatter, kLow>, dim3(blocks), dim3(QWARPS * 32), 0, stream,
                    static_cast<const __nv_bfloat16*>(src), gather, gather_div, scatter, n_copies, n_rows, K,
                    static_cast<uint8_t*>(q), s, wide, kept, n_routed);
}

cudaError_t launch_quant_planes(const void* src, int64_t n_rows, int K, void* q, float* s, bool four_bit, int32_t* wide,
                                const int32_t* kept, int64_t n_routed, cudaStream_t stream) {
    auto launch = four_bit ? launch_quant<true, false, kLowBits> : launch_quant<false, false, kLowBits>;
    return launch(src, nullptr, 1, nullptr, 1, n_rows, K, q, s, wide, kept, n_routed, stream);
}

cudaError_t launch_quant_rows(const void* src, const int32_t* gather, int gather_div, int64_t n_rows, int K, void* q,
                              float* s, cudaStream_t stream) {
    return launch_quant<false, false, 0>(src, gather, gather_div, nullptr, 1, n_rows, K, q, s, nullptr, nullptr, 0, stream);
}

// 2048 tokens x 8 copies, H 7168: 45 us, against 86 quantising each of the
// 16384 gathered rows (every one a full read and all the arithmetic again).
cudaError_t launch_quant_scatter(const void* src, const int32_t* pair_pos, int k, int64_t n_src, int K, void* q, float* s,
                                 cudaStream_t stream) {
    return launch_quant<false, true, 0>(src, nullptr, 1, pair_pos, k, n_src, K, q, s, nullptr, nullptr, 0, stream);
}

}  // namespace gbmoe
