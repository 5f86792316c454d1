// MoE Gate: router logits, expert choice and routing weights.
//
// Two kernels. gate_logits computes l[t,e] = x[t,:].Wg[e,:] (+ bias[e]) in
// fp32 in the fixed order the layer's definition uses (32 partial sums over
// interleaved 8-element chunks, one fused multiply-add per element, then a
// butterfly of pairwise sums), so the expert choice is bit-identical to the
// oracle's. A warp owns TB tokens x EB experts; lane l holds the partial sums
// of chunks l, l+32, ... for all of them, which is exactly the fixed order.
// select_experts then runs one warp per token over the logits. Large batches
// use a shared-memory-staged variant with the same order (below).
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "kernels.h"

namespace gbmoe {

constexpr int kGateWarps = 8;

// A small batch is bound by the latency of a warp's H / 256 dependent steps:
// the loads of U steps are in flight together, and small warp tiles spread the
// work over more SMs (their repeated reads come from L2).
// A warp's logits of rows t0 .. of x and experts e0 ..
template <typename TA, int TB, int EB, int U>
__device__ __forceinline__ void gate_logits_warp(const TA* __restrict__ x, const TA* __restrict__ wg,
                                                 const float* __restrict__ bias, float* __restrict__ logits, int t0,
                                                 int e0, int T, int H, int E) {
    const int lane = threadIdx.x & 31;
    float acc[TB][EB];
    const TA* xp[TB];  // rows past the end repeat the last one and are not stored
    const TA* wp[EB];
#pragma unroll
    for (int a = 0; a < TB; ++a) xp[a] = x + (size_t)min(t0 + a, T - 1) * H + 8 * lane;
#pragma unroll
    for (int b = 0; b < EB; ++b) wp[b] = wg + (size_t)min(e0 + b, E - 1) * H + 8 * lane;
#pragma unroll
    for (int a = 0; a < TB; ++a)
#pragma unroll
        for (int b = 0; b < EB; ++b) acc[a][b] = 0.0f;

    const int steps = H / 256;  // H % 256 == 0: a lane's chunks are lane, lane + 32, ..
    for (int s0 = 0; s0 < steps; s0 += U) {
        Raw8<TA> xr[U][TB], wr[U][EB];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (s0 + u >= steps) break;
#pragma unroll
            for (int a = 0; a < TB; ++a) xr[u][a].load(xp[a] + 256 * (s0 + u));
#pragma unroll
            for (int b = 0; b < EB; ++b) wr[u][b].load(wp[b] + 256 * (s0 + u));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (s0 + u >= steps) break;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int a = 0; a < TB; ++a)
#pragma unroll
                    for (int b = 0; b < EB; ++b) acc[a][b] = __fmaf_rn(xr[u][a].at(i), wr[u][b].at(i), acc[a][b]);
        }
    }
    // butterfly: s[p] <- s[p] + s[p ^ d], d = 16 .. 1 (one commutative add: all lanes end equal)
#pragma unroll
    for (int a = 0; a < TB; ++a)
#pragma unroll
        for (int b = 0; b < EB; ++b) {
            float v = acc[a][b];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, d));
            acc[a][b] = v;
        }
#pragma unroll
    for (int a = 0; a < TB; ++a)
#pragma unroll
        for (int b = 0; b < EB; ++b) {
            const int t = t0 + a, e = e0 + b;
            if (lane == a * EB + b && t < T && e < E) {
                float l = acc[a][b];
                if (bias) l = __fadd_rn(l, bias[e]);
                logits[(size_t)t * E + e] = l;
            }
        }
}

template <typename TA, int TB, int EB, int U>
__global__ void __launch_bounds__(kGateWarps * 32)
gate_logits_kernel(const TA* __restrict__ x, const TA* __restrict__ wg, const float* __restrict__ bias,
                   float* __restrict__ logits, int T, int H, int E) {
    pdl_enter();
    const int e0 = (blockIdx.y * kGateWarps + (threadIdx.x >> 5)) * EB;
    if (e0 < E) gate_logits_warp<TA, TB, EB, U>(x, wg, bias, logits, blockIdx.x * TB, e0, T, H, E);
}

template <typename TA, int TB, int EB, int U>
static cudaError_t launch_gate_logits(const TA* x, const TA* wg, const float* bias, float* logits, int T, int H, int E,
                                      cudaStream_t stream) {
    const dim3 grid((unsigned)((T + TB - 1) / TB), (unsigned)((E + kGateWarps * EB - 1) / (kGateWarps * EB)));
    return launch_k(gate_logits_kernel<TA, TB, EB, U>, grid, dim3(kGateWarps * 32), 0, stream, x, wg, bias, logits, T, H,
                    E);
}

// Warp tiles by batch: few tokens leave most SMs idle unless a warp takes few
// experts; more tokens make the rows' repeated L2 reads the cost.
template <typename TA>
static cudaError_t launch_gate_logits(const TA* x, const TA* wg, const float* bias, float* logits, int T, int H, int E,
                                      cudaStream_t stream) {
    constexpr int U = 8 / sizeof(TA);  // 4 steps of bf16, 2 of fp32
    if (T <= 4) return launch_gate_logits<TA, 1, 2, 2 * U>(x, wg, bias, logits, T, H, E, stream);
    if (T <= 64) return launch_gate_logits<TA, 2, 4, U>(x, wg, bias, logits, T, H, E, stream);
    return launch_gate_logits<TA, 4, 4, U / 2>(x, wg, bias, logits, T, H, E, stream);
}

// Large batches: the same fixed order, as a CUDA-core GEMM. A CTA owns 32
// tokens x 16 experts; 256-element slabs of x and Wg go through a
// cp.async ring in shared memory, and warp w (of 8) accumulates tokens
// 8*(w%4).. x experts 8*(w/4).. in registers. Lane l reads 8-element chunk l
// of every slab, i.e. chunks l, l+32, ... in increasing order, elements in
// increasing order inside a chunk, exactly as in the definition.
constexpr int kGT = 32, kGE = 16, kSlab = 256, kGStages = 3;
constexpr size_t kGateTiledSmem = (size_t)kGStages * (kGT + kGE) * kSlab * 2;

__device__ __forceinline__ void cp_async_16_or_zero(void* dst, const void* src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const int n = valid ? 16 : 0;  // 0 bytes read: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// With a token list, tile rows are the listed tokens (list[0 .. *n_list)), and
// tiles past the list's end return at once, as all do when the list is short
// enough for gate_logits_list_kernel.
constexpr int kShortList = 128;
__global__ void __launch_bounds__(256, 1)
gate_logits_tiled_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ wg,
                         const float* __restrict__ bias, float* __restrict__ logits, int T, int H, int E,
                         const int32_t* __restrict__ list, const int32_t* __restrict__ n_list) {
    pdl_enter();
    const int n_rows = list ? *n_list : T;
    if (list && n_rows <= kShortList) return;
    if ((int)blockIdx.x * kGT >= n_rows) return;
    // token of tile row i (or -1 past the end)
    auto token = [&](int i) -> int {
        const int r = (int)blockIdx.x * kGT + i;
        return r < n_rows ? (list ? list[r] : r) : -1;
    };
    extern __shared__ __align__(16) uint8_t smem[];
    uint8_t* sx = smem;                                          // [stage][kGT][kSlab] bf16
    uint8_t* sw = smem + (size_t)kGStages * kGT * kSlab * 2;     // [stage][kGE][kSlab] bf16
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e0 = blockIdx.y * kGE;
    const int nslab = H / kSlab;

    // thread i copies chunk i % 32 of rows i / 32 + 8 m of a slab (kGT rows of
    // x, then kGE of Wg): their sources are looked up once, not per slab (the
    // flagged tokens of 2048 x 256, H 7168: 83 -> 61 us)
    constexpr int kRows = (kGT + kGE) / 8;
    const __nv_bfloat16* src[kRows];
    bool ok[kRows];
#pragma unroll
    for (int m = 0; m < kRows; ++m) {
        const int row = warp + 8 * m;
        if (row < kGT) {
            const int t = token(row);
            ok[m] = t >= 0;
            src[m] = x + (size_t)(ok[m] ? t : 0) * H + 8 * lane;
        } else {
            const int e = e0 + row - kGT;
            ok[m] = e < E;
            src[m] = wg + (size_t)(ok[m] ? e : 0) * H + 8 * lane;
        }
    }
    auto load_slab = [&](int j) {
        const int st = j % kGStages;
#pragma unroll
        for (int m = 0; m < kRows; ++m) {
            const int row = warp + 8 * m;
            uint8_t* dst = row < kGT ? sx + ((size_t)st * kGT + row) * kSlab * 2 : sw + ((size_t)st * kGE + row - kGT) * kSlab * 2;
            cp_async_16_or_zero(dst + 16 * lane, src[m] + (size_t)j * kSlab, ok[m]);
        }
    };

    float acc[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.0f;
    const int tg = (warp & 3) * 8, eg = (warp >> 2) * 8;

#pragma unroll
    for (int j = 0; j < kGStages - 1; ++j) {
        if (j < nslab) load_slab(j);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int j = 0; j < nslab; ++j) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGStages - 2) : "memory");
        __syncthreads();
        if (j + kGStages - 1 < nslab) load_slab(j + kGStages - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const int st = j % kGStages;
        uint4 xr[8], wr[8];
#pragma unroll
        for (int a = 0; a < 8; ++a)
            xr[a] = *reinterpret_cast<const uint4*>(sx + (((size_t)st * kGT + tg + a) * kSlab + 8 * lane) * 2);
#pragma unroll
        for (int b = 0; b < 8; ++b)
            wr[b] = *reinterpret_cast<const uint4*>(sw + (((size_t)st * kGE + eg + b) * kSlab + 8 * lane) * 2);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float xf[8], wf[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const uint32_t u = (&xr[a].x)[i >> 1];
                xf[a] = (i & 1) ? bf16hi(u) : bf16lo(u);
            }
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const uint32_t u = (&wr[b].x)[i >> 1];
                wf[b] = (i & 1) ? bf16hi(u) : bf16lo(u);
            }
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 8; ++b) acc[a][b] = __fmaf_rn(xf[a], wf[b], acc[a][b]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // butterfly: s[p] <- s[p] + s[p ^ d], d = 16 .. 1
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            float v = acc[a][b];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, d));
            acc[a][b] = v;
        }
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int t = token(tg + a), e = e0 + eg + b;
            if (lane == ((a * 8 + b) & 31) && t >= 0 && e < E) {
                float l = acc[a][b];
                if (bias) l = __fadd_rn(l, bias[e]);
                logits[(size_t)t * E + e] = l;
            }
        }
}

// The listed tokens' logits when the list is short (the audit flags a few
// tokens per thousand; the tiled kernel above then keeps a handful of CTAs
// waiting through H / 256 slabs: 26 us for a handful of tokens at H 4096, 6.6
// here). Longer lists are the tiled kernel's.
constexpr int kListBlocks = 32;

__global__ void __launch_bounds__(kGateWarps * 32)
gate_logits_list_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ wg,
                        const float* __restrict__ bias, float* __restrict__ logits, int T, int H, int E,
                        const int32_t* __restrict__ list, const int32_t* __restrict__ n_list) {
    pdl_enter();
    const int n = *n_list;
    const int e0 = (blockIdx.y * kGateWarps + (threadIdx.x >> 5)) * 2;
    if (n > kShortList || e0 >= E) return;
    for (int i = blockIdx.x; i < n; i += kListBlocks)
        gate_logits_warp<__nv_bfloat16, 1, 2, 8>(x, wg, bias, logits, list[i], e0, T, H, E);
}

// ------------------------------------------------------- expert choice

// Fixed fp32 exponential for the sigmoid score (the expert choice depends on
// its exact bits, so it is not left to a library): NaN is returned as it
// is, anything else clamped to [-86, 88];
// n = rint(x*log2 e); r = (x - n*ln2_hi) - n*ln2_lo with ln2_hi the leading
// 16 bits of ln 2 (Cody-Waite reduction, exact n*ln2_hi); exp(r) from its
// degree-8 Taylor polynomial by Horner's rule, a separate rounded multiply
// and add per step; times 2^n assembled from exponent bits.
__device__ __forceinline__ float pinned_exp(float x) {
    const float kLog2e = __uint_as_float(0x3fb8aa3bu);  // fp32(1/ln 2)
    const float kLn2Hi = __uint_as_float(0x3f317200u);  // 0.693145751953125
    const float kLn2Lo = __uint_as_float(0x35bfbe8eu);  // fp32(ln 2 - kLn2Hi)
    const uint32_t kInvFact[9] = {0x3f800000u, 0x3f800000u, 0x3f000000u, 0x3e2aaaabu, 0x3d2aaaabu,
                                  0x3c088889u, 0x3ab60b61u, 0x39500d01u, 0x37d00d01u};  // fp32(1/i!)
    if (x != x) return x;  // NaN in, NaN out
    x = fminf(fmaxf(x, -86.0f), 88.0f);
    float n = rintf(__fmul_rn(x, kLog2e));
    float r = __fsub_rn(x, __fmul_rn(n, kLn2Hi));
    r = __fsub_rn(r, __fmul_rn(n, kLn2Lo));
    float p = __uint_as_float(kInvFact[8]);
#pragma unroll
    for (int i = 7; i >= 0; --i) p = __fadd_rn(__fmul_rn(p, r), __uint_as_float(kInvFact[i]));
    return __fmul_rn(p, __uint_as_float((uint32_t)((int)n + 127) << 23));
}

__device__ __forceinline__ float pinned_sigmoid(float l) {
    return __fdiv_rn(1.0f, __fadd_rn(1.0f, pinned_exp(-l)));
}

constexpr int kNone = 0x7fffffff;  // the index of no candidate

// Key a score takes in the expert choice: a NaN counts as -infinity, so
// non-finite logits still give valid, deterministic ids (ties to the lower index).
__device__ __forceinline__ float choice_key(float v) { return v != v ? -INFINITY : v; }

// A key as an unsigned integer of the same order (both zeros alike), above 0
// for every real candidate, so that the warp's best is one redux each for the
// key and the index.
__device__ __forceinline__ uint32_t key_bits(float k) {
    const uint32_t u = __float_as_uint(k == 0.0f ? 0.0f : k);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t b) {
    return __uint_as_float(b ^ ((b >> 31) ? 0x80000000u : 0xffffffffu));
}

// the best (largest key, then smallest index) of the lanes' candidates; a lane
// without one has key bits 0 and index kNone
__device__ __forceinline__ void warp_best(uint32_t& kb, int& i) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, kb);
    i = __reduce_min_sync(0xffffffffu, kb == m ? i : kNone);
    kb = m;
}

constexpr int kSelWarps = 4;

// Audit of router logits computed on the tensor cores (their fp32 sums run in
// the hardware's own order, not the fixed order of the definition). Those
// logits differ from the fixed-order ones by at most about
// scale * ||x_t|| * ||w_e|| (|sum of the same products in two orders|), so an
// expert choice whose every deciding comparison clears twice that bound is the
// fixed-order choice; any other token is recomputed in the fixed order.
struct GateAudit {
    const __nv_bfloat16* x;   // [T, H]; null: logits are fixed-order already (no audit)
    const float* wnorm_max;   // max_e ||wg[e]||_2 (one float)
    float scale;              // bound on |tensor-core logit - fixed-order logit| / (||x_t|| * max ||w_e||)
    int32_t* flagged;         // [T] tokens whose choice is too close to call (their logits are recomputed)
    int32_t* n_flagged;       // their count
};

// Where a logit is still in parts: the sum of n planes, stride floats apart,
// plus bias (n = 1 and no bias: it is complete).
struct LogitPlanes {
    int n;
    int64_t stride;
    const float* bias;
};

// Chooses token t's experts and weights, by one warp: lane j < k returns slot
// j's expert in sel_id and weight in w. Expert e lives in lane e % 32, register
// e / 32 (E <= 32 * SLOTS); key and val are this warp's shared arrays of E
// floats (choice keys; logits or sigmoids).
template <int SLOTS>
__device__ __forceinline__ void select_token(const float* __restrict__ l, const LogitPlanes& pl, const float* __restrict__ select_bias,
                                             const RouteParams& rp, const GateAudit& au, int t, float* key, float* val,
                                             int& sel_id, float& w) {
    const int lane = threadIdx.x & 31;
    const int E = rp.E, k = rp.top_k;
    const bool sigmoid = rp.score == GBMOE_SIGMOID;
    const int G = sigmoid ? rp.n_group : 1;
    const int gs = E / G;
    float raw[SLOTS];
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) raw[s] = lane + 32 * s < E ? l[lane + 32 * s] : 0.0f;
    for (int q = 1; q < pl.n; ++q) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
            if (lane + 32 * s < E) raw[s] = __fadd_rn(raw[s], l[q * pl.stride + lane + 32 * s]);
    }
    if (pl.bias) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
            if (lane + 32 * s < E) raw[s] = __fadd_rn(raw[s], pl.bias[lane + 32 * s]);
    }
    uint32_t kb[SLOTS];  // candidates: 0 once chosen, or not allowed
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
        const int e = lane + 32 * s;
        kb[s] = 0;
        if (e < E) {
            float v = raw[s];
            if (sigmoid) {
                v = pinned_sigmoid(v);
                val[e] = v;
                if (select_bias) v = __fadd_rn(v, select_bias[e]);
            } else {
                val[e] = v;
            }
            v = choice_key(v);
            kb[s] = key_bits(v);
            if (G > 1) key[e] = v;
        }
    }
    __syncwarp();

    // groups kept (bit g set); all experts allowed without group limiting.
    // margin_g: gap between the last kept and the best dropped group score
    float margin_g = INFINITY;
    if (G > 1) {
        // the two largest q of each group: 32 / G lanes share a group's
        // experts when G divides the warp, else one lane takes them all
        const int L = 32 % G == 0 ? 32 / G : 1;
        const int g = lane / L;
        float a = -INFINITY, b = -INFINITY;
        if (g < G)
            for (int e = g * gs + lane % L; e < (g + 1) * gs; e += L) {
                const float v = key[e];
                if (v > a) { b = a; a = v; } else if (v > b) { b = v; }
            }
        for (int d = 1; d < L; d <<= 1) {
            const float ao = __shfl_xor_sync(0xffffffffu, a, d), bo = __shfl_xor_sync(0xffffffffu, b, d);
            b = fmaxf(fminf(a, ao), fmaxf(b, bo));
            a = fmaxf(a, ao);
        }
        const float gscore = choice_key(__fadd_rn(a, b));  // inf + -inf is NaN
        // one candidate per group, in the group's first lane
        uint32_t gb = g < G && lane % L == 0 ? key_bits(gscore) : 0u;
        uint32_t kept = 0u;
        float last = 0.0f;
        for (int r = 0; r <= rp.topk_group && r < G; ++r) {
            uint32_t m = gb;
            int ii = gb ? g : kNone;
            warp_best(m, ii);
            if (r == rp.topk_group) {  // the best dropped group
                margin_g = last - key_value(m);
                break;
            }
            kept |= 1u << (ii & 31);  // topk_group <= G groups hold candidates
            if (g == ii) gb = 0u;
            last = key_value(m);
        }
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
            if (!((kept >> (((lane + 32 * s) / gs) & 31)) & 1u)) kb[s] = 0u;
    }

    // top-k over allowed experts, descending key, ties to the lower index;
    // margin_k: smallest gap between consecutive keys of the k chosen and
    // the best one left out
    sel_id = 0;
    float top_key = 0.0f, prev = 0.0f, margin_k = INFINITY;
    for (int j = 0; j <= k; ++j) {
        uint32_t m = 0u;
        int ii = kNone;
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
            if (kb[s] > m) { m = kb[s]; ii = lane + 32 * s; }
        warp_best(m, ii);
        const bool found = ii < E;
        const float kk = found ? key_value(m) : -INFINITY;
        if (j > 0 && found) margin_k = fminf(margin_k, prev - kk);
        if (j == k) break;  // only the margin to the best expert left out
        // found always (check_config keeps top_k within the kept groups' experts)
#pragma unroll
        for (int s = 0; s < SLOTS; ++s)
            if (ii == lane + 32 * s) kb[s] = 0u;
        if (j == 0) top_key = kk;
        if (lane == j) sel_id = found ? ii : 0;
        prev = kk;
    }

    if (au.x) {
        // bound on the logit error, and on the key error it causes (sigmoid:
        // slope <= 1/4, plus a few units in the last place of the fp32 key)
        float xx = 0.0f;
        const __nv_bfloat16* xt = au.x + (size_t)t * rp.H;
        for (int c0 = lane; c0 < rp.H / 8; c0 += 4 * 32) {
            Raw8<__nv_bfloat16> xv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c0 + 32 * u < rp.H / 8) xv[u].load(xt + 8 * (c0 + 32 * u));
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c0 + 32 * u < rp.H / 8) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) xx = fmaf(xv[u].at(i), xv[u].at(i), xx);
                }
        }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) xx += __shfl_xor_sync(0xffffffffu, xx, d);
        // (plus a few units in the last place of the logits, for the bias add)
        const float bl = au.scale * sqrtf(xx) * *au.wnorm_max + 1e-6f * (1.0f + fabsf(top_key));
        const float bk = sigmoid ? 0.25f * bl + 1e-6f : bl;
        const bool close = !(margin_k > 2.0f * bk) || !(margin_g > 4.0f * bk);
        if (close && lane == 0) au.flagged[atomicAdd(au.n_flagged, 1)] = t;
    }

    // routing weights (lane j < k holds slot j)
    w = 0.0f;
    if (!sigmoid) {
        float lj = (lane < k) ? val[sel_id] : 0.0f;
        float m = top_key, z = 0.0f;
        if (!rp.renormalize) {
            float mm = -INFINITY;
#pragma unroll
            for (int s = 0; s < SLOTS; ++s)
                if (lane + 32 * s < E) mm = fmaxf(mm, raw[s]);
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, d));
            m = mm;
#pragma unroll
            for (int s = 0; s < SLOTS; ++s)
                if (lane + 32 * s < E) z += expf(raw[s] - m);
        } else {
            z = (lane < k) ? expf(lj - m) : 0.0f;
        }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) z += __shfl_xor_sync(0xffffffffu, z, d);
        w = (lane < k) ? expf(lj - m) / z * rp.routed_scale : 0.0f;
    } else {
        float sj = (lane < k) ? val[sel_id] : 0.0f;
        float z = sj;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) z += __shfl_xor_sync(0xffffffffu, z, d);
        w = (rp.renormalize ? sj / z : sj) * rp.routed_scale;
    }
    __syncwarp();
}

// One warp per token (every token, or those of `list` in grid-stride order).
template <int SLOTS>
__global__ void __launch_bounds__(kSelWarps * 32)
select_experts_kernel(const float* __restrict__ logits, LogitPlanes pl, const float* __restrict__ select_bias,
                      int32_t* __restrict__ topk_ids, float* __restrict__ topk_w, RouteParams rp, GateAudit au,
                      const int32_t* __restrict__ list, const int32_t* __restrict__ n_list) {
    pdl_enter();
    __shared__ float s_key[kSelWarps][32 * SLOTS];
    __shared__ float s_val[kSelWarps][32 * SLOTS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_tok = list ? *n_list : rp.T;
    for (int i = blockIdx.x * kSelWarps + warp; i < n_tok; i += gridDim.x * kSelWarps) {
        const int t = list ? list[i] : i;
        int id;
        float w;
        select_token<SLOTS>(logits + (size_t)t * rp.E, pl, select_bias, rp, au, t, s_key[warp], s_val[warp], id, w);
        if (lane < rp.top_k) {
            topk_ids[(size_t)t * rp.top_k + lane] = id;
            topk_w[(size_t)t * rp.top_k + lane] = w;
        }
    }
}

static cudaError_t launch_select(const float* logits, const LogitPlanes& pl, const float* select_bias, int32_t* topk_ids, float* topk_w,
                                 const RouteParams& rp, const GateAudit& au, const int32_t* list, const int32_t* n_list,
                                 int blocks, cudaStream_t stream) {
    auto kernel = rp.E <= 128 ? select_experts_kernel<4> : rp.E <= 256 ? select_experts_kernel<8> : select_experts_kernel<16>;
    return launch_k(kernel, dim3(blocks), dim3(kSelWarps * 32), 0, stream, logits, pl, select_bias, topk_ids, topk_w, rp, au,
                    list, n_list);
}

// max over experts of ||wg[e]||_2 (fp32) into *out (zeroed beforehand): a
// warp per router row; the maximum taken on the float bits, which order like
// the values for non-negative floats
__global__ void __launch_bounds__(256)
row_norm_max_kernel(const __nv_bfloat16* __restrict__ wg, int E, int H, float* __restrict__ out) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int e = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (e >= E) return;
    float ss = 0.0f;
    for (int c = lane; c < H / 8; c += 32) {
        float v[8];
        Vec8<__nv_bfloat16>::load(wg + (size_t)e * H + 8 * c, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) ss = fmaf(v[i], v[i], ss);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
    if (lane == 0) atomicMax(reinterpret_cast<int*>(out), __float_as_int(sqrtf(ss)));
}

// Bound on |tensor-core logit - fixed-order logit| / (||x_t|| * max_e ||w_e||)
// that the audit uses (from measured differences on the workloads, with a
// safety factor; GBMOE_GATE_AUDIT_SCALE overrides it for tests).
constexpr float kGateAuditScale = 2.0e-6f;

static float gate_audit_scale() {
    const char* v = std::getenv("GBMOE_GATE_AUDIT_SCALE");
    if (!v || !*v) return kGateAuditScale;
    char* end = nullptr;
    const float f = std::strtof(v, &end);
    return (end != v && *end == '\0' && f >= 0.0f) ? f : kGateAuditScale;
}

// The tiled gate kernel over the whole batch, or over a list of its tokens.
static cudaError_t launch_gate_tiled(const void* x, const void* wg, const float* bias, float* logits, int T, int H, int E,
                                     const int32_t* list, const int32_t* n_list, cudaStream_t stream) {
    static DeviceOnce smem_set;  // shared-memory size, set once per device
    const cudaError_t e = smem_set.run([] {
        return cudaFuncSetAttribute(gate_logits_tiled_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kGateTiledSmem);
    });
    if (e != cudaSuccess) return e;
    const dim3 grid((T + kGT - 1) / kGT, (E + kGE - 1) / kGE);  // (tiles past a list's end exit)
    return launch_k(gate_logits_tiled_kernel, grid, dim3(256), kGateTiledSmem, stream,
                    static_cast<const __nv_bfloat16*>(x), static_cast<const __nv_bfloat16*>(wg), bias, logits, T, H, E,
                    list, n_list);
}

// ------------------------------------------------ RMSNorm before the gate

// y = x / sqrt(mean(x^2) + eps) * gamma per row, in the order of the gate's
// logits (its output decides the routing): one warp per row; lane l takes
// the 8-element chunks l, l+32, ... and sums their squares with one fused
// multiply-add each; the 32 partial sums are combined by the butterfly of
// pairwise additions; then ms = ss / H, v = ms + eps, r = sqrt(v), inv = 1 / r
// and y = (x * inv) * gamma, every step one correctly rounded fp32
// operation; y is rounded once to the activation type.
template <typename TA>
__global__ void __launch_bounds__(256)
rmsnorm_kernel(const TA* __restrict__ x, const TA* __restrict__ gamma, float eps, int T, int H, TA* __restrict__ y) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (t >= T) return;
    const TA* xr = x + t * H;
    float ss = 0.0f;
    for (int c = lane; c < H / 8; c += 32) {
        float v[8];
        Vec8<TA>::load(xr + 8 * c, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) ss = __fmaf_rn(v[i], v[i], ss);
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xffffffffu, ss, d));
    const float ms = __fdiv_rn(ss, (float)H);
    const float inv = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(ms, eps)));
    for (int c = lane; c < H / 8; c += 32) {
        float v[8], g[8], o[8];
        Vec8<TA>::load(xr + 8 * c, v);
        Vec8<TA>::load(gamma + 8 * c, g);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = __fmul_rn(__fmul_rn(v[i], inv), g[i]);
        Vec8<TA>::store(y + t * H + 8 * c, o);
    }
}

cudaError_t launch_rmsnorm(const void* x, const void* gamma, float eps, int T, int H, int act_dtype, void* y,
                           cudaStream_t stream) {
    if (T == 0) return cudaSuccess;
    const dim3 grid((unsigned)((T + 7) / 8));
    cudaError_t le;
    if (act_dtype == GBMOE_BF16)
        le = launch_k(rmsnorm_kernel<__nv_bfloat16>, grid, dim3(256), 0, stream, static_cast<const __nv_bfloat16*>(x),
                      static_cast<const __nv_bfloat16*>(gamma), eps, T, H, static_cast<__nv_bfloat16*>(y));
    else
        le = launch_k(rmsnorm_kernel<float>, grid, dim3(256), 0, stream, static_cast<const float*>(x),
                      static_cast<const float*>(gamma), eps, T, H, static_cast<float*>(y));
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

cudaError_t launch_route(const RouteParams& rp, const void* x, const void* wg, const float* logit_bias,
                         const float* select_bias, float* logits, int32_t* topk_ids, float* topk_w,
                         const RouteScratch& rs, cudaStream_t stream) {
    if (rp.T == 0) return cudaSuccess;
    GateAudit au{};
    if (rp.gate_tc) {
        // tensor-core logits, then the audited choice
        auto xp = static_cast<const __nv_bfloat16*>(x);
        auto wp = static_cast<const __nv_bfloat16*>(wg);
        if (const cudaError_t me = cudaMemsetAsync(rs.audit, 0, 8, stream); me != cudaSuccess)  // norm max, count
            return me;
        if (const cudaError_t le = launch_k(row_norm_max_kernel, dim3((rp.E + 7) / 8), dim3(256), 0, stream, wp,
                rp.E, rp.H, rs.audit); le != cudaSuccess)
            return le;
        if (const cudaError_t le = launch_gate_tc(x, wg, logits, rp.T, rp.H, rp.E, rs.sched, rs.err,
                stream); le != cudaSuccess)
            return le;
        au.x = xp; au.wnorm_max = rs.audit; au.scale = gate_audit_scale();
        au.flagged = rs.flagged; au.n_flagged = reinterpret_cast<int32_t*>(rs.audit + 1);
    } else if (rp.act_dtype == GBMOE_BF16) {
        auto xp = static_cast<const __nv_bfloat16*>(x);
        auto wp = static_cast<const __nv_bfloat16*>(wg);
        if (rp.T >= 1024) {
            if (const cudaError_t le = launch_gate_tiled(x, wg, logit_bias, logits, rp.T, rp.H, rp.E, nullptr,
                    nullptr, stream); le != cudaSuccess)
                return le;
        } else if (const cudaError_t le = launch_gate_logits(xp, wp, logit_bias, logits, rp.T, rp.H, rp.E, stream);
                   le != cudaSuccess) {
            return le;
        }
    } else {
        if (const cudaError_t le = launch_gate_logits(static_cast<const float*>(x), static_cast<const float*>(wg),
                logit_bias, logits, rp.T, rp.H, rp.E, stream); le != cudaSuccess)
            return le;
    }
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    const LogitPlanes whole{1, 0, nullptr};
    const LogitPlanes parts{rp.gate_tc ? gate_tc_splits(rp.T, rp.H, rp.E) : 1, (int64_t)rp.T * rp.E, logit_bias};
    if ((err = launch_select(logits, rp.gate_tc ? parts : whole, select_bias, topk_ids, topk_w, rp, au, nullptr, nullptr,
                             (rp.T + kSelWarps - 1) / kSelWarps, stream)) != cudaSuccess || !rp.gate_tc)
        return err;
    // flagged tokens: fixed-order logits, then their choice again (no audit)
    const int32_t* n_flag = reinterpret_cast<const int32_t*>(rs.audit + 1);
    const int32_t* flagged = rs.flagged;
    if ((err = launch_k(gate_logits_list_kernel,
                        dim3(std::min(rp.T, kListBlocks), (rp.E + 2 * kGateWarps - 1) / (2 * kGateWarps)),
                        dim3(kGateWarps * 32), 0, stream, static_cast<const __nv_bfloat16*>(x),
                        static_cast<const __nv_bfloat16*>(wg), logit_bias, logits, rp.T, rp.H, rp.E, flagged,
                        n_flag)) != cudaSuccess)
        return err;
    if ((err = launch_gate_tiled(x, wg, logit_bias, logits, rp.T, rp.H, rp.E, flagged, n_flag, stream)) !=
        cudaSuccess)
        return err;
    const GateAudit none{};
    return launch_select(logits, whole, select_bias, topk_ids, topk_w, rp, none, flagged, n_flag, sm_count() * 4, stream);
}

}  // namespace gbmoe
