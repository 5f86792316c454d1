// Fused MoE on CUDA cores: tiled grouped GEMMs in fp32.
//
// The route for fp32 activations (where tensor-core inputs would lose the
// fp32 precision the layer is specified in) and for any weight format. A CTA
// of 128 threads computes BM rows of one expert x 128 weight rows (stage 1: 64
// gate rows and the 64 up rows of the same columns, then h = silu(g) * u;
// stage 2: 128 down rows); a thread holds BM / 8 rows x 8 columns, four of
// them 64 weight rows after the other four, so that gate and up of a column
// meet in one thread. Slabs of 16 k go through two shared buffers, k-major;
// the next slab's global loads are in flight while the current one is
// multiplied, weights are decoded to fp32 as they are stored. Every sum runs
// over k in order with one fused multiply-add per product.
//
// Bound by fp32 FMA issue: pairs of columns share one instruction
// (fma.rn.f32x2), and 8 x 8 outputs take 4 16-byte shared loads per k where
// 2 x 2 took 6 scalar ones. 1001 tokens, top 4 of 16 experts, H 1024, I 768,
// fp32: gate/up 578 -> 304 us (41 TFLOP/s), down 351 -> 166 us; same bits.
#include "common.cuh"
#include "ffn_sched.h"
#include "kernels.h"
#include "wload.cuh"

namespace gbmoe {

constexpr int kBN = 128, kBK = 16;
constexpr int kSimtThreads = 128;
constexpr int kPad = 4;

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Eight consecutive weights of a row as stored, and their decoding: the bytes
// of element k0 (a multiple of 8) on, and the scale that covers it.
template <int WQ>
struct Load8 {
    static constexpr int WORDS = WQ == GBMOE_F32 ? 8 : WQ == GBMOE_BF16 ? 4 : WQ == GBMOE_FP8_E4M3_B128 ? 2 : 1;
    uint32_t w[WORDS];
    float sc;
    __device__ __forceinline__ void load(const void* base, const void* scales, int64_t e, int N, int K, int n, int k0) {
        const int64_t at = ((e * N + n) * K + k0) * WORDS / 8;  // in words
        const uint32_t* p = static_cast<const uint32_t*>(base) + at;
        if constexpr (WORDS >= 4) {
#pragma unroll
            for (int i = 0; i < WORDS / 4; ++i) {
                const uint4 v = ld_stream16(p + 4 * i);
                w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
            }
        } else if constexpr (WORDS == 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(p);
            w[0] = v.x; w[1] = v.y;
        } else {
            w[0] = p[0];
        }
        if constexpr (WORDS <= 2) sc = WFmt<WQ>::scale(scales, e, N, K, n, k0);
    }
    __device__ __forceinline__ void decode(float (&v)[8]) const {
        if constexpr (WQ == GBMOE_F32) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(w[i]);
        } else if constexpr (WQ == GBMOE_BF16) {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = i & 1 ? bf16hi(w[i >> 1]) : bf16lo(w[i >> 1]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if constexpr (WQ == GBMOE_FP8_E4M3_B128) v[i] = e4m3_to_f32((w[i >> 2] >> (8 * (i & 3))) & 0xffu) * sc;
                else if constexpr (WQ == GBMOE_INT4_G128) v[i] = int4_to_f32((w[0] >> (4 * i)) & 0xfu) * sc;
                else v[i] = e2m1_to_f32((w[0] >> (4 * i)) & 0xfu) * sc;
            }
        }
    }
};

template <int WQ, int STAGE>
__device__ __forceinline__ const void* w_base(const FfnProblem& p, int half) {
    return STAGE == 2 ? p.w_down : half ? p.w_up : p.w_gate;
}
template <int WQ, int STAGE>
__device__ __forceinline__ const void* w_scales(const FfnProblem& p, int half) {
    return STAGE == 2 ? p.s_down : half ? p.s_up : p.s_gate;
}

template <typename TA, int WQ, int STAGE, int BM>
__global__ void __launch_bounds__(kSimtThreads, BM == 64 ? 4 : 5)
simt_gemm_kernel(FfnProblem p) {
    pdl_enter();
    constexpr int TM = BM / 8;              // rows of a thread
    constexpr int A_GROUPS = BM * 2;        // 8-element pieces of a slab's rows
    __shared__ __align__(16) float As[2][kBK][BM + kPad];
    __shared__ __align__(16) float Bs[2][kBK][kBN + kPad];
    __shared__ int32_t s_src[BM];
    const int32_t* sched = p.sched;
    const int tile = blockIdx.x;
    if (tile >= sched[1]) return;
    const int2 tl = reinterpret_cast<const int2*>(sched + sched_tiles_offset(p.E))[tile];
    const int e = tl.x;
    const int64_t cnt = p.counts ? p.counts[e] : p.n_rows;
    const int64_t row0 = (p.offsets ? p.offsets[e] : 0) + (int64_t)tl.y * BM;
    const int rows = (int)min64(BM, cnt - (int64_t)tl.y * BM);
    const int K = STAGE == 1 ? p.H : p.I, N = STAGE == 1 ? p.I : p.H;
    const int n0 = blockIdx.y * (STAGE == 1 ? kBN / 2 : kBN);
    const int t = threadIdx.x;
    if (t < BM) {
        const int64_t r = row0 + t;
        int32_t src = -1;
        if (t < rows) src = STAGE == 1 && p.sorted_pair ? p.sorted_pair[r] / p.pair_div : (int32_t)r;
        s_src[t] = src;
    }
    __syncthreads();
    const TA* a = static_cast<const TA*>(STAGE == 1 ? p.x : p.h);

    // thread t loads piece t % 2 (8 k) of row t / 2 of A and of each 64-row half of B
    const int lrow = t >> 1, lk = 8 * (t & 1);
    const bool loads_a = t < A_GROUPS;
    const int src = loads_a ? s_src[lrow] : -1;
    const TA* a_src = a + (int64_t)(src >= 0 ? src : 0) * K + lk;
    float av[8];
    Load8<WQ> bv[2];
    auto load = [&](int k0) {
        if (src >= 0) {
            Vec8<TA>::load(a_src + k0, av);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) av[i] = 0.0f;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            bv[h].load(w_base<WQ, STAGE>(p, h), w_scales<WQ, STAGE>(p, h), e, N, K, n0 + lrow + (STAGE == 2 ? 64 * h : 0),
                       k0 + lk);
    };
    auto store = [&](int buf) {
        if (loads_a) {
#pragma unroll
            for (int i = 0; i < 8; ++i) As[buf][lk + i][lrow] = av[i];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[8];
            bv[h].decode(v);
#pragma unroll
            for (int i = 0; i < 8; ++i) Bs[buf][lk + i][64 * h + lrow] = v[i];
        }
    };

    const int tx = t & 15, ty = t >> 4;
    uint64_t acc[TM][4];  // column pairs: 4 tx + {0, 1}, {2, 3}, then the same 64 columns on
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;
    load(0);
    store(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < K; k0 += kBK, buf ^= 1) {
        if (k0 + kBK < K) load(k0 + kBK);
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            float ar[TM];
#pragma unroll
            for (int i = 0; i < TM; i += 4)
                *reinterpret_cast<float4*>(&ar[i]) = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM + i]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][4 * tx]);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][64 + 4 * tx]);
            const uint64_t b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const uint64_t aa = pack2(ar[i], ar[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(aa, b[j], acc[i][j]);
            }
        }
        if (k0 + kBK < K) store(buf ^ 1);
        __syncthreads();
    }

    TA* out = static_cast<TA*>(STAGE == 1 ? p.h : p.y);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = ty * TM + i;
        if (r >= rows) break;
        TA* o = out + (row0 + r) * N + n0 + 4 * tx;
        const float2 c0 = unpack2(acc[i][0]), c1 = unpack2(acc[i][1]), c2 = unpack2(acc[i][2]), c3 = unpack2(acc[i][3]);
        if constexpr (STAGE == 1) {
            o[0] = from_f32<TA>(silu_mul(c0.x, c2.x));
            o[1] = from_f32<TA>(silu_mul(c0.y, c2.y));
            o[2] = from_f32<TA>(silu_mul(c1.x, c3.x));
            o[3] = from_f32<TA>(silu_mul(c1.y, c3.y));
        } else {
            o[0] = from_f32<TA>(c0.x); o[1] = from_f32<TA>(c0.y); o[2] = from_f32<TA>(c1.x); o[3] = from_f32<TA>(c1.y);
            o[64] = from_f32<TA>(c2.x); o[65] = from_f32<TA>(c2.y); o[66] = from_f32<TA>(c3.x); o[67] = from_f32<TA>(c3.y);
        }
    }
}

template <typename TA, int WQ, int BM>
static cudaError_t launch_simt_bm(const FfnProblem& p, cudaStream_t stream) {
    cudaError_t err = launch_ffn_schedule(p.counts, p.E, p.n_rows, BM, p.sched, stream);
    if (err != cudaSuccess) return err;
    const unsigned max_tiles = (unsigned)sched_max_tiles(p.E, p.n_rows, BM);
    if ((err = launch_k(simt_gemm_kernel<TA, WQ, 1, BM>, dim3(max_tiles, p.I / (kBN / 2)), dim3(kSimtThreads), 0, stream,
                        p)) != cudaSuccess)
        return err;
    return launch_k(simt_gemm_kernel<TA, WQ, 2, BM>, dim3(max_tiles, p.H / kBN), dim3(kSimtThreads), 0, stream, p);
}

// 64-row tiles reuse each weight slab twice as often; up to 40 rows per expert
// most experts fill one 32-row tile or two
template <typename TA, int WQ>
static cudaError_t launch_simt_t(const FfnProblem& p, cudaStream_t stream) {
    if (p.n_rows == 0) return cudaSuccess;
    return p.n_rows <= 40 * (int64_t)p.E ? launch_simt_bm<TA, WQ, 32>(p, stream) : launch_simt_bm<TA, WQ, 64>(p, stream);
}

cudaError_t launch_ffn_simt(const FfnProblem& p, cudaStream_t stream) {
    if (p.act_dtype == GBMOE_BF16) {
        switch (p.w_dtype) {
            case GBMOE_F32: return launch_simt_t<__nv_bfloat16, GBMOE_F32>(p, stream);
            case GBMOE_BF16: return launch_simt_t<__nv_bfloat16, GBMOE_BF16>(p, stream);
            case GBMOE_FP8_E4M3_B128: return launch_simt_t<__nv_bfloat16, GBMOE_FP8_E4M3_B128>(p, stream);
            case GBMOE_INT4_G128: return launch_simt_t<__nv_bfloat16, GBMOE_INT4_G128>(p, stream);
            case GBMOE_MXFP4: return launch_simt_t<__nv_bfloat16, GBMOE_MXFP4>(p, stream);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (p.w_dtype) {
        case GBMOE_F32: return launch_simt_t<float, GBMOE_F32>(p, stream);
        case GBMOE_BF16: return launch_simt_t<float, GBMOE_BF16>(p, stream);
        case GBMOE_FP8_E4M3_B128: return launch_simt_t<float, GBMOE_FP8_E4M3_B128>(p, stream);
        case GBMOE_INT4_G128: return launch_simt_t<float, GBMOE_INT4_G128>(p, stream);
        case GBMOE_MXFP4: return launch_simt_t<float, GBMOE_MXFP4>(p, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gbmoe
