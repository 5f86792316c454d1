// Fused MoE for few rows per expert (decode): weight streaming.
//
// With ~2 rows per expert the layer is bound by reading each active expert's
// weights once from HBM. Each CTA takes one active expert and a slice of
// output columns; its warps stream weight rows with 16-byte non-allocating
// loads (four 16-byte chunks of each of its 4 rows in flight per lane: 8 KB per
// warp) and dot them against the expert's activation rows, which sit in
// shared memory. Lane l takes the 16-byte chunks l, l+32, ... of a row, so a
// warp reads 512 contiguous bytes per row and step. The inner loop reloads
// each activation chunk once and decodes the weights per activation row, so
// the kernel stays within 128 registers and two CTAs (16 warps) share an SM.
// Up to kNT rows are handled per weight pass; more rows take further passes
// over the same weights. A CTA covers up to 4 column groups in turn, so it
// stages its activation rows once for all of them.
//   stage 1: h[r, i] = silu(x_r . Wgate[i]) * (x_r . Wup[i]), 2 columns per warp
//   stage 2: y[r, n] = h_r . Wdown[n], 4 output columns per warp
#pragma once

#include <type_traits>

#include "common.cuh"
#include "ffn_sched.h"
#include "kernels.h"
#include "wload.cuh"

namespace gbmoe {

constexpr int kStreamWarps = 8;
constexpr int kNT = 8;      // activation rows per weight pass
constexpr int kMaxGroupsPerCta = 4;
constexpr int kMinWaves = 8;

// CTAs per SM the register budget is set for: two for plain weights (fp32: kTwo,
// see two_ctas); quantised ones decode more per element and get the whole register
// file
template <int WQ, bool kTwo>
constexpr int stream_min_blocks() { return WQ == GBMOE_BF16 || (WQ == GBMOE_F32 && kTwo) ? 2 : 1; }

// 8-element (or 16-byte) chunks of a row loaded before use. fp32: two of 32 bytes
// fit 128 registers, so two CTAs share an SM; with four one CTA took it alone
// (tiny fp32 layer: gate/up 17.2 -> 12.0 us, the passes apart as well, see
// passes_apart; 4 tokens of 16 experts, H 1024, I 768: layer 56 -> 42 us).
template <int WQ, bool kTwo>
constexpr int kUnroll = WQ == GBMOE_F32 && kTwo ? 2 : 4;

// acc[q][r] += W_q . xs[r] for 4 weight rows q (byte pointers wrow, scale rows
// srow) and NT activation rows r in shared memory (row stride K).
template <typename TA, int WQ, int NT, bool kTwo>
__device__ __forceinline__ void dot4(const uint8_t* const (&wrow)[4], const void* const (&srow)[4], const TA* xs,
                                     int K, float (&acc)[4][NT]) {
    using F = WFmt<WQ>;
    const int lane = threadIdx.x & 31;
    const int nchunk = K / F::CE;
    constexpr int CB = F::NV * 16;  // bytes per chunk
    constexpr int U = kUnroll<WQ, kTwo>;
    for (int c0 = lane; c0 < nchunk; c0 += 32 * U) {
        uint4 raw[U][4][F::NV];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + 32 * u;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int v = 0; v < F::NV; ++v)
                    raw[u][q][v] = c < nchunk ? ld_stream16(wrow[q] + (size_t)c * CB + 16 * v) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + 32 * u;
            if (c >= nchunk) break;
            float sc[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) sc[q] = F::scale_at(srow[q], c * F::CE);
#pragma unroll
            for (int sub = 0; sub < F::CE / 8; ++sub) {
                const int k0 = c * F::CE + 8 * sub;
#pragma unroll
                for (int r = 0; r < NT; ++r) {
                    float xv[8];
                    Vec8<TA>::load(xs + (size_t)r * K + k0, xv);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float w[8];
                        F::decode8(raw[u][q], sub, sc[q], w);
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[q][r] = fmaf(w[i], xv[i], acc[q][r]);
                    }
                }
            }
        }
    }
}

// Sums of the 4 * NT partial sums over the warp, each the same tree as a
// butterfly over d = 16 .. 1, but halving the values a lane carries at each step
// (31 shuffles for 32 values, not 160): lane l returns the sum of value
// l >> (5 - log2(4 * NT)), value q * NT + r being acc[q][r].
template <int NT>
__device__ __forceinline__ float warp_sums(const float (&acc)[4][NT]) {
    constexpr int V = 4 * NT;
    const int lane = threadIdx.x & 31;
    float v[V];
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = acc[i / NT][i % NT];
#pragma unroll
    for (int n = V / 2, d = 16; d >= 1; d >>= 1, n >>= 1) {
        if (n >= 1) {
            const bool upper = lane & d;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const float keep = upper ? v[i + n] : v[i], give = upper ? v[i] : v[i + n];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, d);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
        }
    }
    return v[0];
}

// Copies nt activation rows into shared memory: row r is source row
// sorted_pair[row0 + r] / pair_div (row0 + r itself without sorted_pair).
template <typename TA>
__device__ void stage_rows(TA* xs, const TA* src, int K, const int32_t* sorted_pair, int pair_div, int64_t row0,
                           int nt) {
    const int per_row = K * (int)sizeof(TA) / 16;
    for (int idx = threadIdx.x; idx < nt * per_row; idx += blockDim.x) {
        const int r = idx / per_row, c = idx % per_row;
        int64_t srow = row0 + r;
        if (sorted_pair) srow = sorted_pair[srow] / pair_div;
        reinterpret_cast<uint4*>(xs + (size_t)r * K)[c] = reinterpret_cast<const uint4*>(src + srow * K)[c];
    }
}

template <typename F>
__device__ __forceinline__ void dispatch_nt(int nt, F&& f) {
    if (nt <= 1) f(std::integral_constant<int, 1>{});
    else if (nt <= 2) f(std::integral_constant<int, 2>{});
    else if (nt <= 4) f(std::integral_constant<int, 4>{});
    else f(std::integral_constant<int, 8>{});
}

// Weight rows of column group g: 2 gate + 2 up rows (stage 1) or 4 down rows
// (stage 2) per warp, with their scale rows; col0 = first output column.
template <int WQ, int STAGE>
__device__ __forceinline__ void group_rows(const FfnProblem& p, int e, int g, int warp, const uint8_t* (&wrow)[4],
                                           const void* (&srow)[4], int& col0) {
    using F = WFmt<WQ>;
    const int H = p.H, I = p.I;
    if (STAGE == 1) {
        const size_t rb = F::row_bytes(H);
        const int i0 = (g * kStreamWarps + warp) * 2;
        const uint8_t* wg = static_cast<const uint8_t*>(p.w_gate) + (size_t)e * I * rb;
        const uint8_t* wu = static_cast<const uint8_t*>(p.w_up) + (size_t)e * I * rb;
        wrow[0] = wg + i0 * rb; wrow[1] = wg + (i0 + 1) * rb; wrow[2] = wu + i0 * rb; wrow[3] = wu + (i0 + 1) * rb;
        srow[0] = F::scale_row(p.s_gate, e, I, H, i0); srow[1] = F::scale_row(p.s_gate, e, I, H, i0 + 1);
        srow[2] = F::scale_row(p.s_up, e, I, H, i0); srow[3] = F::scale_row(p.s_up, e, I, H, i0 + 1);
        col0 = i0;
    } else {
        const size_t rb = F::row_bytes(I);
        const int n0 = (g * kStreamWarps + warp) * 4;
        const uint8_t* wd = static_cast<const uint8_t*>(p.w_down) + (size_t)e * H * rb;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            wrow[q] = wd + (n0 + q) * rb;
            srow[q] = F::scale_row(p.s_down, e, H, I, n0 + q);
        }
        col0 = n0;
    }
}

// One CTA: one active expert and gpc consecutive column groups (a group is 8
// warps x 2 h-columns in stage 1, 8 warps x 4 y-columns in stage 2). The
// expert's activation rows are staged once per pass of kNT rows and serve
// all of the CTA's groups.
//   stage 1: h[r, i] = silu(x_r . Wgate[i]) * (x_r . Wup[i])
//   stage 2: y[r, n] = h_r . Wdown[n]
template <typename TA, int WQ, int STAGE, bool kTwo>
__device__ __forceinline__ void stream_ffn_cta(const FfnProblem& p, int gpc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TA* xs = reinterpret_cast<TA*>(smem_raw);
    const int slot = blockIdx.x;
    if (slot >= p.sched[0]) return;
    const int e = p.sched[kSchedHeader + slot];
    const int64_t cnt = p.counts ? p.counts[e] : p.n_rows;
    const int64_t row0 = p.offsets ? p.offsets[e] : 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = STAGE == 1 ? p.H : p.I;
    TA* out = static_cast<TA*>(STAGE == 1 ? p.h : p.y);
    const int out_cols = STAGE == 1 ? p.I : p.H;
    for (int64_t p0 = (int64_t)blockIdx.z * kNT; p0 < cnt; p0 += (int64_t)gridDim.z * kNT) {
        const int nt = (int)min64(kNT, cnt - p0);
        __syncthreads();
        if (STAGE == 1) stage_rows<TA>(xs, static_cast<const TA*>(p.x), K, p.sorted_pair, p.pair_div, row0 + p0, nt);
        else stage_rows<TA>(xs, static_cast<const TA*>(p.h), K, nullptr, 1, row0 + p0, nt);
        __syncthreads();
        dispatch_nt(nt, [&](auto NTc) {
            constexpr int NT = decltype(NTc)::value;
#pragma unroll 1
            for (int g = blockIdx.y * gpc; g < (blockIdx.y + 1) * gpc; ++g) {
                const uint8_t* wrow[4];
                const void* srow[4];
                int col0;
                group_rows<WQ, STAGE>(p, e, g, warp, wrow, srow, col0);
                float acc[4][NT];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int r = 0; r < NT; ++r) acc[q][r] = 0.0f;
                dot4<TA, WQ, NT, kTwo>(wrow, srow, xs, K, acc);
                const float sum = warp_sums<NT>(acc);
                constexpr int COPIES = 8 / NT;  // lanes that hold the same sum
                const int value = lane / COPIES, q = value / NT, r = value % NT;
                TA* dst = out + (row0 + p0 + r) * out_cols + col0;
                if (STAGE == 1) {  // q 0, 1: gate; the up sums are 16 lanes on
                    const float up = __shfl_xor_sync(0xffffffffu, sum, 16);
                    if (q < 2 && r < nt && lane % COPIES == 0) dst[q] = from_f32<TA>(silu_mul(sum, up));
                } else if (r < nt && lane % COPIES == 0) {
                    dst[q] = from_f32<TA>(sum);
                }
            }
        });
    }
}

template <typename TA, int WQ, bool kTwo>
__global__ void __launch_bounds__(kStreamWarps * 32, stream_min_blocks<WQ, kTwo>())
stream_gateup_kernel(FfnProblem p, int gpc) {
    pdl_enter();
    stream_ffn_cta<TA, WQ, 1, kTwo>(p, gpc);
}

template <typename TA, int WQ, bool kTwo>
__global__ void __launch_bounds__(kStreamWarps * 32, stream_min_blocks<WQ, kTwo>())
stream_down_kernel(FfnProblem p, int gpc) {
    pdl_enter();
    stream_ffn_cta<TA, WQ, 2, kTwo>(p, gpc);
}

// Column groups per CTA: up to kMaxGroupsPerCta while the grid keeps at least
// kMinWaves waves of CTAs (fewer, longer CTAs stage the rows less often;
// too few CTAs leave SMs idle). groups is a multiple of 8.
inline int groups_per_cta(int max_active, int groups) {
    const int64_t slots = (int64_t)sm_count() * 2;  // resident CTAs (two per SM)
    int gpc = kMaxGroupsPerCta;
    while (gpc > 1 && (int64_t)max_active * (groups / gpc) < kMinWaves * slots) gpc /= 2;
    return gpc;
}

// Passes of kNT rows that run side by side, in CTAs of their own: as many as an
// expert has on average, while the grid does not fill the SMs (the weights of
// such a grid stay in L2, so reading them again costs less than waiting).
inline int passes_apart(int64_t n_rows, int max_active, int ctas) {
    const int64_t avg = (n_rows + (int64_t)max_active * kNT - 1) / ((int64_t)max_active * kNT);
    int z = 1;
    while (2 * z <= avg && (int64_t)ctas * z < (int64_t)sm_count() * 2) z *= 2;
    return z;
}

// fp32: whether two CTAs share an SM: where the grid has a second one for it, and
// where the rows of both leave the L1 cache room for the loads in flight (16 experts,
// top 4, H 3584, 12 tokens: layer 337 us with both CTAs' 112 KB of rows, 263 with one
// CTA and four chunks; H 3072, 96 KB each: 146 and 156).
inline bool two_ctas(int64_t ctas, size_t smem) { return ctas > sm_count() && smem <= 96 * 1024; }

template <typename TA, int WQ, bool kTwo>
static cudaError_t launch_stream_gateup(const FfnProblem& p, dim3 grid, size_t smem, int gpc, cudaStream_t stream) {
    static DeviceOnce smem_set;  // the most dynamic shared memory any problem may ask for, set once per device
    const cudaError_t err = smem_set.run([] {
        return cudaFuncSetAttribute(stream_gateup_kernel<TA, WQ, kTwo>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)stream_smem_budget());
    });
    if (err != cudaSuccess) return err;
    return launch_k(stream_gateup_kernel<TA, WQ, kTwo>, grid, dim3(kStreamWarps * 32), smem, stream, p, gpc);
}

template <typename TA, int WQ, bool kTwo>
static cudaError_t launch_stream_down(const FfnProblem& p, dim3 grid, size_t smem, int gpc, cudaStream_t stream) {
    static DeviceOnce smem_set;
    const cudaError_t err = smem_set.run([] {
        return cudaFuncSetAttribute(stream_down_kernel<TA, WQ, kTwo>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)stream_smem_budget());
    });
    if (err != cudaSuccess) return err;
    return launch_k(stream_down_kernel<TA, WQ, kTwo>, grid, dim3(kStreamWarps * 32), smem, stream, p, gpc);
}

template <typename TA, int WQ>
static cudaError_t launch_stream_t(const FfnProblem& p, cudaStream_t stream) {
    const int max_active = (int)min64(p.E, p.n_rows);
    if (max_active == 0) return cudaSuccess;
    const size_t smem1 = (size_t)kNT * p.H * sizeof(TA);
    const size_t smem2 = (size_t)kNT * p.I * sizeof(TA);
    const int groups1 = p.I / (2 * kStreamWarps), groups2 = p.H / (4 * kStreamWarps);
    const int gpc1 = groups_per_cta(max_active, groups1), gpc2 = groups_per_cta(max_active, groups2);
    dim3 g1(max_active, groups1 / gpc1), g2(max_active, groups2 / gpc2);
    g1.z = passes_apart(p.n_rows, max_active, g1.x * g1.y);
    g2.z = passes_apart(p.n_rows, max_active, g2.x * g2.y);
    // (other formats have one variant)
    constexpr bool kOne = WQ == GBMOE_F32;
    auto two = [](const dim3& g, size_t smem) { return !kOne || two_ctas((int64_t)g.x * g.y * g.z, smem); };
    const cudaError_t err = two(g1, smem1) ? launch_stream_gateup<TA, WQ, true>(p, g1, smem1, gpc1, stream)
                                           : launch_stream_gateup<TA, WQ, !kOne>(p, g1, smem1, gpc1, stream);
    if (err != cudaSuccess) return err;
    return two(g2, smem2) ? launch_stream_down<TA, WQ, true>(p, g2, smem2, gpc2, stream)
                          : launch_stream_down<TA, WQ, !kOne>(p, g2, smem2, gpc2, stream);
}

// launch_stream_t for one weight format, defined in ffn_stream_<format>.cu so
// that the formats' kernel instantiations compile in parallel
template <int WQ>
cudaError_t launch_stream_w(const FfnProblem& p, cudaStream_t stream);
// int4 weights with fp32 activations (ffn_stream_int4w_f32a.cu)
cudaError_t launch_stream_int4w_f32a(const FfnProblem& p, cudaStream_t stream);

}  // namespace gbmoe
