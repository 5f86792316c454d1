// Fused MoE on CUDA cores: tiled grouped GEMMs in fp32.
//
// The route for fp32 activations (where tensor-core inputs would lose the
// fp32 precision the layer is specified in) and for any weight format. A CTA
// of 128 threads computes BM rows of one expert x BN weight rows (stage 1: BN / 2
// gate rows and the up rows of the same columns, then h = silu(g) * u; stage 2:
// BN down rows); a thread holds BM / 8 rows x BN / 16 columns, half of them BN / 2
// weight rows after the others, so that gate and up of a column meet in one
// thread. Slabs of 2048 / BN k go through two shared buffers, k-major; the next
// slab's global loads are in flight while the current one is multiplied, weights
// are decoded to fp32 as they are stored. Every sum runs over k in order with one
// fused multiply-add per product, whatever the tile.
//
// Large grids are bound by fp32 FMA issue: pairs of columns share one
// instruction (fma.rn.f32x2), and 8 x 8 outputs take 4 16-byte shared loads per k
// where 2 x 2 took 6 scalar ones. 1001 tokens, top 4 of 16 experts, H 1024, I 768,
// fp32: gate/up 578 -> 304 us (41 TFLOP/s), down 351 -> 166 us; same bits. Small
// ones are bound by a CTA's walk over k, a load's latency per slab: BN 64 gives
// twice the CTAs half the slabs. 70 tokens, one expert, H 3840, I 128, int4: layer
// 309 -> 131 us (2 x 2 outputs and a slab without prefetch: 242).
#include "common.cuh"
#include "ffn_sched.h"
#include "kernels.h"
#include "wload.cuh"

namespace gbmoe {

constexpr int kSimtThreads = 128;
constexpr int kPad = 4;

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

template <typename TA, int WQ, int STAGE, int BM, int BN>
__global__ void __launch_bounds__(kSimtThreads, BM == 64 ? 4 : 5)
simt_gemm_kernel(FfnProblem p) {
    pdl_enter();
    constexpr int kBK = 2048 / BN;          // k of a slab
    constexpr int PIECES = kBK / 8;         // 8-element pieces of a slab's row
    constexpr int HALF = BN / 2;            // gate and up rows, or the down rows' two halves
    constexpr int TM = BM / 8;              // rows of a thread
    constexpr int PAIRS = BN / 64;          // column pairs of a thread in each half
    __shared__ __align__(16) float As[2][kBK][BM + kPad];
    __shared__ __align__(16) float Bs[2][kBK][BN + kPad];
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
    const int n0 = blockIdx.y * (STAGE == 1 ? HALF : BN);
    const int t = threadIdx.x;
    if (t < BM) {
        const int64_t r = row0 + t;
        int32_t src = -1;
        if (t < rows) src = STAGE == 1 && p.sorted_pair ? p.sorted_pair[r] / p.pair_div : (int32_t)r;
        s_src[t] = src;
    }
    __syncthreads();
    const TA* a = static_cast<const TA*>(STAGE == 1 ? p.x : p.h);

    // thread t loads piece t % PIECES of row t / PIECES of each half of B, and of A
    // (the rows HALF on too where A has them)
    const int lrow = t / PIECES, lk = 8 * (t % PIECES);
    constexpr int A_LOADS = BM > HALF ? BM / HALF : 1;
    const bool loads_a = lrow < BM;
    int src[A_LOADS];
    const TA* a_src[A_LOADS];
#pragma unroll
    for (int i = 0; i < A_LOADS; ++i) {
        src[i] = loads_a ? s_src[lrow + HALF * i] : -1;
        a_src[i] = a + (int64_t)(src[i] >= 0 ? src[i] : 0) * K + lk;
    }
    float av[A_LOADS][8];
    Load8<WQ> bv[2];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < A_LOADS; ++i) {
            if (src[i] >= 0) {
                Vec8<TA>::load(a_src[i] + k0, av[i]);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) av[i][j] = 0.0f;
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            bv[h].load(w_base<WQ, STAGE>(p, h), w_scales<WQ, STAGE>(p, h), e, N, K, n0 + lrow + (STAGE == 2 ? HALF * h : 0),
                       k0 + lk);
    };
    auto store = [&](int buf) {
        if (loads_a) {
#pragma unroll
            for (int i = 0; i < A_LOADS; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) As[buf][lk + j][lrow + HALF * i] = av[i][j];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v[8];
            bv[h].decode(v);
#pragma unroll
            for (int i = 0; i < 8; ++i) Bs[buf][lk + i][HALF * h + lrow] = v[i];
        }
    };

    const int tx = t & 15, ty = t >> 4;
    uint64_t acc[TM][2 * PAIRS];  // column pairs 2 (PAIRS tx + j), then the same HALF columns on
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 2 * PAIRS; ++j) acc[i][j] = 0;
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
            uint64_t b[2 * PAIRS];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float* bp = &Bs[buf][kk][HALF * h + 2 * PAIRS * tx];
                if constexpr (PAIRS == 2) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(bp);
                    b[2 * h] = v.x;
                    b[2 * h + 1] = v.y;
                } else {
                    b[h] = *reinterpret_cast<const uint64_t*>(bp);
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const uint64_t aa = pack2(ar[i], ar[i]);
#pragma unroll
                for (int j = 0; j < 2 * PAIRS; ++j) acc[i][j] = fma2(aa, b[j], acc[i][j]);
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
        TA* o = out + (row0 + r) * N + n0 + 2 * PAIRS * tx;
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) {
            const float2 lo = unpack2(acc[i][j]), hi = unpack2(acc[i][PAIRS + j]);
            if constexpr (STAGE == 1) {
                o[2 * j] = from_f32<TA>(silu_mul(lo.x, hi.x));
                o[2 * j + 1] = from_f32<TA>(silu_mul(lo.y, hi.y));
            } else {
                o[2 * j] = from_f32<TA>(lo.x);
                o[2 * j + 1] = from_f32<TA>(lo.y);
                o[HALF + 2 * j] = from_f32<TA>(hi.x);
                o[HALF + 2 * j + 1] = from_f32<TA>(hi.y);
            }
        }
    }
}

template <typename TA, int WQ, int STAGE, int BM, int BN>
static cudaError_t launch_simt_gemm(const FfnProblem& p, cudaStream_t stream) {
    const unsigned cols = STAGE == 1 ? p.I / (BN / 2) : p.H / BN;
    return launch_k(simt_gemm_kernel<TA, WQ, STAGE, BM, BN>, dim3((unsigned)sched_max_tiles(p.E, p.n_rows, BM), cols),
                    dim3(kSimtThreads), 0, stream, p);
}

// 64-row tiles reuse each weight slab twice as often; up to 40 rows per expert
// most experts fill one 32-row tile or two, and a problem that has neither stage
// fill the SMs twice with 64-row tiles of 128 weight rows is better off with more,
// smaller ones. A stage takes 64 weight rows per CTA where 128 would leave SMs
// with fewer CTAs than run side by side on one (5 of 32 rows; 3 of 64). 146 problems
// from 17 to 24000 rows, fp32 activations, all formats, geometric mean over the
// 32 x 32 tiles of 2 x 2 outputs: 1.31 with 128 weight rows everywhere (0.78 at
// worst), 1.61 with 32 x 64 tiles everywhere, 1.67 with this rule (1.01 at worst).
constexpr int64_t kTallCtasPerSm = 2, kNarrowTallCtasPerSm = 3, kNarrowCtasPerSm = 5;

template <typename TA, int WQ>
static cudaError_t launch_simt_t(const FfnProblem& p, cudaStream_t stream) {
    if (p.n_rows == 0) return cudaSuccess;
    // row tiles there are at least (one per expert with rows, whose number is taken for E at most)
    auto ctas = [&](int stage, int bm) {
        const int64_t tiles = max64((p.n_rows + bm - 1) / bm, min64(p.E, p.n_rows));
        return tiles * (stage == 1 ? p.I / 64 : p.H / 128);
    };
    const int64_t sms = sm_count();
    const bool tall = p.n_rows > 40 * (int64_t)p.E && max64(ctas(1, 64), ctas(2, 64)) >= kTallCtasPerSm * sms;
    cudaError_t err = launch_ffn_schedule(p.counts, p.E, p.n_rows, tall ? 64 : 32, p.sched, stream);
    if (err != cudaSuccess) return err;
    if (tall) {
        err = ctas(1, 64) < kNarrowTallCtasPerSm * sms ? launch_simt_gemm<TA, WQ, 1, 64, 64>(p, stream) : launch_simt_gemm<TA, WQ, 1, 64, 128>(p, stream);
        if (err != cudaSuccess) return err;
        return ctas(2, 64) < kNarrowTallCtasPerSm * sms ? launch_simt_gemm<TA, WQ, 2, 64, 64>(p, stream) : launch_simt_gemm<TA, WQ, 2, 64, 128>(p, stream);
    }
    err = ctas(1, 32) < kNarrowCtasPerSm * sms ? launch_simt_gemm<TA, WQ, 1, 32, 64>(p, stream) : launch_simt_gemm<TA, WQ, 1, 32, 128>(p, stream);
    if (err != cudaSuccess) return err;
    return ctas(2, 32) < kNarrowCtasPerSm * sms ? launch_simt_gemm<TA, WQ, 2, 32, 64>(p, stream) : launch_simt_gemm<TA, WQ, 2, 32, 128>(p, stream);
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
