// Fused MoE, feature-major: quantised weights as the M operand of tcgen05.mma.
//
// With few rows per expert (decode, prefill chunks) a grouped GEMM is bound
// by reading each active expert's weights once. The row-major GEMMs spend a
// 128-row MMA (and its reads of shared memory) on whatever rows the expert
// has; the streaming kernels decode every weight on the CUDA cores once per
// row. Here the weights are the M operand (128 weight rows per MMA, used as
// stored or nearly so) and the expert's rows are the N operand, N rounded to
// the rows that exist, so both the tensor work and the promotion below shrink
// with the rows and the weights' way from HBM to the tensor core is left as
// the bound.
//
// Activations enter as two e4m3 codes per value with one power-of-two scale
// per row and 128 consecutive k, bf16's 8 significant bits in full
// (quant_act.cu).
// Products of codes accumulate in fp32 in tensor memory over 128 k, then the
// promotion warps add the partial sum times its scales to fp32 accumulators
// in registers.
//
//   quant_rows     x (every token once) -> codes and scales
//   gate/up GEMM   -> h = silu(gate) * up (bf16); quant_rows of h
//   down GEMM      -> y (bf16)
//
// One persistent CTA per SM walks (row tile, 256 weight rows) items. Warps:
//   0       TMA of the weight tile of each k block (2 x 128 rows x 128 k),
//           128-byte swizzled, into a ring of stages;
//   1       TMEM (three partial sums) and the MMAs: per k block and 128-row
//           half, q1 and q2 side by side (N = 2 * rows);
//   2-3     gather the row codes with cp.async (the token's row of x, so no
//           sorted copy exists) and their scales;
//   4-11    promotion and the output: warp w reads TMEM lanes 32 * (w % 4)..
//           (weight rows); the rows' groups of 8 alternate between the two sets of
//           four warps.
// A gate/up item holds 128 gate rows and the 128 up rows of the same columns,
// so one thread ends up with gate and up of its column and SwiGLU needs no
// exchange. Every mbarrier wait is bounded (tc_ptx.cuh).
//
// Measured, fp8, 48 tokens, top 8 of 256 experts, H 7168, I 2048 (about 2 rows
// per expert, 8.8 GB of weights): gate/up 1826 -> 767 us and down 1052 -> 397
// us against the streaming kernels, 7.5 TB/s; the layer 3121 -> 1347 us. What
// held it back on the way, per 128-wide k block: waits as calls (2400 -> 1750
// cycles once inlined) and MMAs issued under `lane == 0` (1750 -> 1500).
#include "common.cuh"
#include "ffn_sched.h"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace gbmoe {
namespace fm {

using namespace tc;

constexpr int MB = 128;                 // weight rows per MMA
constexpr int BK = 128;                 // k per block: one swizzle row, one activation scale
constexpr int A_BYTES = 2 * MB * BK;    // the two 128-row halves of an item's weight tile
constexpr int MAX_ROWS = 80;            // most rows of a row tile
constexpr int SLOTS = 3;                // partial sums in TMEM
constexpr int SLOT_COLS = 2 * MAX_ROWS;
constexpr int TMEM_COLS = 512;          // (an allocation is a power of two)
constexpr int MAX_STAGES = 6;
// Scale blocks, used in turn (stages + 2 of them): a block's k block k is
// written once the MMAs of k - stages are done, which were issued once the
// partial sums of k - stages - 2 had been promoted (TMEM holds fewer than two
// k blocks), so the block's last contents have been read by then.
constexpr int RING = MAX_STAGES + 2;
constexpr int SETS = 2;                 // of four promotion warps
constexpr int PROMOTE_WARPS = 4 * SETS;
constexpr int GROUPS = (MAX_ROWS / 8 + SETS - 1) / SETS;  // most groups of 8 rows of a promotion warp
constexpr int GATHER_WARPS = 2;
constexpr int THREADS = 32 * (2 + GATHER_WARPS + PROMOTE_WARPS);
constexpr int NUM_BARS = 3 * MAX_STAGES + 2 * SLOTS + RING + 1;
constexpr int FIXED_BYTES = 1024 + RING * MAX_ROWS * 4 + NUM_BARS * 8 + 16;
constexpr int SMEM_BUDGET = 232448;

constexpr int stage_bytes(int tile_rows) { return A_BYTES + 2 * tile_rows * BK; }
constexpr int stages_for(int tile_rows) {
    const int n = (SMEM_BUDGET - FIXED_BYTES) / stage_bytes(tile_rows);
    return n < MAX_STAGES ? n : MAX_STAGES;
}
static_assert(stages_for(MAX_ROWS) >= 3 && SLOTS <= 4 && SLOTS * SLOT_COLS <= TMEM_COLS, "ring depth");

struct Params {
    int K, n_tiles, out_cols;
    int w_rows_per_expert;  // rows of the weight tensor per expert
    int tile_rows;          // rows of a row tile of the work list (a multiple of 16, at most MAX_ROWS)
    const int32_t* counts;
    const int32_t* offsets;
    const int32_t* sched;
    int E;
    int64_t n_rows;
    __nv_bfloat16* out;
    int32_t* err;
    const uint8_t* q;        // code planes q1, q2: [2][plane_rows][K]
    int64_t plane_rows;
    const float* a_scale;    // [plane_rows][K/128]
    const int32_t* gather;   // row r of the sorted order is plane row gather[r] / gather_div; null: r itself
    int gather_div;
    const float* w_scale0;   // fp8: [E, w_rows_per_expert/128, K/128], first / second half of the item
    const float* w_scale1;
    uint64_t wait_limit_ns;
};

struct Work {
    int e, nt;
    int64_t row0;  // first row of the tile
    int rows;      // rows in the tile
};

__device__ __forceinline__ Work decode_work(const Params& p, int w) {
    const int2* tiles = reinterpret_cast<const int2*>(p.sched + sched_tiles_offset(p.E));
    const int mt = w / p.n_tiles;
    Work r;
    r.nt = w - mt * p.n_tiles;
    const int2 t = tiles[mt];
    r.e = t.x;
    const int64_t cnt = p.counts ? p.counts[t.x] : p.n_rows;
    const int64_t first = (int64_t)t.y * p.tile_rows;
    r.row0 = (p.offsets ? p.offsets[t.x] : 0) + first;
    r.rows = (int)min64(p.tile_rows, cnt - first);
    return r;
}

// rows of one code plane in the N operand (N = 2 * rows_pad, a multiple of 16)
__device__ __forceinline__ int rows_pad(int rows) { return (rows + 7) & ~7; }

// first weight row (of the stacked [E * rows, K] tensor) of each half of item wk
template <bool SWIGLU>
__device__ __forceinline__ void w_rows(const Params& p, const Work& wk, int& a0, int& a1) {
    a0 = wk.e * p.w_rows_per_expert + wk.nt * (SWIGLU ? MB : 2 * MB);
    a1 = SWIGLU ? a0 : a0 + MB;
}

// kind::f8f6f4, fp32 accumulator, e4m3 x e4m3, K-major, M = 128
__device__ __forceinline__ uint32_t idesc_f8(int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(MB >> 4) << 24); }

__device__ __forceinline__ void mma_f8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void cp_async_16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// ------------------------------- pairs of fp32 (one instruction for two)

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t pack2u(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// 8 columns of this thread's TMEM lane, not waited for
__device__ __forceinline__ void tmem_ld8(uint32_t t, uint32_t (&a)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7])
                 : "r"(t));
}
// the wait for the loads above; their registers pass through it, so that no
// use of them moves above it
__device__ __forceinline__ void tmem_wait(uint32_t (&a)[8], uint32_t (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&a)[8], uint32_t (&b)[8], uint32_t (&c)[8], uint32_t (&d)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]),
                   "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6]), "+r"(c[7]),
                   "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7])
                 :
                 : "memory");
}

// acc += (a + b) * (sc * w) over 8 rows: a, b the q1 and q2 partial sums, sc
// the rows' scales in shared memory, w the weight scale in both halves
__device__ __forceinline__ void promote8(const uint32_t (&a)[8], const uint32_t (&b)[8], const float* sc, uint64_t w,
                                         uint64_t* acc) {
    const float4 f0 = *reinterpret_cast<const float4*>(sc), f1 = *reinterpret_cast<const float4*>(sc + 4);
    const uint64_t f[4] = {pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        acc[i] = fma2(add2(pack2u(a[2 * i], a[2 * i + 1]), pack2u(b[2 * i], b[2 * i + 1])), mul2(f[i], w), acc[i]);
}

// -------------------------------------------------------------- the GEMM

template <bool SWIGLU>
__global__ void __launch_bounds__(THREADS, 1)
fm_gemm_kernel(const __grid_constant__ CUtensorMap tm_w0, const __grid_constant__ CUtensorMap tm_w1, const Params p,
               const int stages) {
    pdl_enter();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int b_bytes = 2 * p.tile_rows * BK;
    uint8_t* sA = smem;
    uint8_t* sB = smem + stages * A_BYTES;
    float* sS = reinterpret_cast<float*>(sB + stages * b_bytes);  // [RING][MAX_ROWS]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sS + RING * MAX_ROWS);
    uint64_t* wfull = bars;                   // weights of a k block landed
    uint64_t* bfull = bars + MAX_STAGES;      // its row codes landed
    uint64_t* empty = bars + 2 * MAX_STAGES;  // MMAs reading the stage finished
    uint64_t* pfull = bars + 3 * MAX_STAGES;  // partial sum ready
    uint64_t* pempty = pfull + SLOTS;         // partial sum read by every promoting warp
    uint64_t* sfull = pempty + SLOTS;         // scale block written
    uint64_t* drain = sfull + RING;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&bfull[s], GATHER_WARPS * 32);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < SLOTS; ++b) {
            mbar_init(&pfull[b], 1);
            mbar_init(&pempty[b], PROMOTE_WARPS);
        }
        for (int b = 0; b < RING; ++b) mbar_init(&sfull[b], GATHER_WARPS);
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int total = p.sched[1] * p.n_tiles;
    const int nkb = p.K / BK;

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------ weight producer
        int stage = 0;
        uint32_t phase = 0;
        uint32_t inflight = 0, inflight_par = 0;  // stages loaded but not seen consumed
        bool ok = true;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            int a0, a1;
            w_rows<SWIGLU>(p, wk, a0, a1);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                inflight &= ~(1u << stage);
                mbar_expect_tx(&wfull[stage], A_BYTES);
                tma_load_2d(sA + stage * A_BYTES, &tm_w0, kb * BK, a0, &wfull[stage]);
                tma_load_2d(sA + stage * A_BYTES + A_BYTES / 2, &tm_w1, kb * BK, a1, &wfull[stage]);
                inflight |= 1u << stage;
                inflight_par = (inflight_par & ~(1u << stage)) | (phase << stage);
                if (++stage == stages) { stage = 0; phase ^= 1; }
            }
        }
        // every copy issued lands before the CTA leaves
        for (int s = 0; s < stages; ++s)
            if ((inflight >> s) & 1u) drain_wait(&wfull[s], (inflight_par >> s) & 1u);
    } else if (warp == 1) {
        // ------------------------- MMA issuer (the whole warp, one lane issues)
        int stage = 0;
        uint32_t phase = 0;
        uint32_t slot = 0, sphase = 0;
        bool ok = true, issued = false;
        const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = __shfl_sync(0xffffffffu, rows_pad(wk.rows), 0);  // warp-uniform
            const uint32_t idesc = idesc_f8(2 * rp);
            for (int kb = 0; kb < nkb; ++kb) {
                if (!warp_wait(&bfull[stage], phase, abort_flag, p.err, p.wait_limit_ns) ||
                    !warp_wait(&wfull[stage], phase, abort_flag, p.err, p.wait_limit_ns)) {
                    ok = false;
                    break;
                }
                // the row codes were written through the generic proxy (cp.async)
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                const uint64_t db = db0 + (uint64_t)(stage * b_bytes >> 4);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (!warp_wait(&pempty[slot], sphase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d = tmem_base + slot * SLOT_COLS;
                    const uint64_t dh = da0 + (uint64_t)((stage * A_BYTES + half * (MB * BK)) >> 4);
                    if (elect_one()) {
#pragma unroll
                        for (int j = 0; j < BK / 32; ++j)  // +32 bytes along K per instruction
                            mma_f8(d, dh + 2 * j, db + 2 * j, idesc, j != 0 ? 1u : 0u);
                        mma_commit(&pfull[slot]);
                        if (half == 1) mma_commit(&empty[stage]);
                    }
                    __syncwarp();
                    issued = true;
                    if (++slot == SLOTS) { slot = 0; sphase ^= 1; }
                }
                if (!ok) break;
                if (++stage == stages) { stage = 0; phase ^= 1; }
            }
        }
        if (issued) {  // every MMA issued has finished before TMEM is released
            if (elect_one()) mma_commit(drain);
            __syncwarp();
            drain_wait(drain, 0);
        }
    } else if (warp >= 2 && warp < 2 + GATHER_WARPS) {
        // ---------------------------------------------- row codes, scales
        // thread t copies 16-byte chunk t % 8 of rows t / 8 + 8 i in both
        // planes (8 whole 128-byte rows per pass of the two warps) and the
        // scales of rows t and t + 64
        const int t = threadIdx.x - 64;
        const int chunk = t & 7, r0 = t >> 3;
        int stage = 0, ring = 0;
        uint32_t phase = 0;
        bool ok = true;
        const int64_t plane = p.plane_rows * p.K;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = rows_pad(wk.rows);
            auto src_row = [&](int j) -> int64_t {  // plane row of tile row j (past the tile's end: any valid row)
                if (j >= wk.rows) return 0;
                const int64_t r = wk.row0 + j;
                if (!p.gather) return r;
                const int32_t g = p.gather[r];
                return g >= 0 ? g / p.gather_div : 0;
            };
            const uint8_t* src[MAX_ROWS / 8];
#pragma unroll
            for (int i = 0; i < MAX_ROWS / 8; ++i) src[i] = p.q + (8 * i < rp ? src_row(r0 + 8 * i) : 0) * p.K + 16 * chunk;
            const float* s0 = p.a_scale + (t < rp ? src_row(t) : 0) * nkb;  // (MAX_ROWS <= 128: two per thread)
            const float* s1 = p.a_scale + (t + 64 < rp ? src_row(t + 64) : 0) * nkb;
            float n0 = s0[0], n1 = s1[0];
            for (int kb = 0; kb < nkb; ++kb) {
                if (!warp_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                uint8_t* dst = sB + stage * b_bytes;
#pragma unroll
                for (int i = 0; i < MAX_ROWS / 8; ++i) {
                    if (8 * i >= rp) break;
                    const uint32_t off = sw128_off(r0 + 8 * i, chunk);
                    cp_async_16(dst + off, src[i] + kb * BK);
                    cp_async_16(dst + rp * BK + off, src[i] + plane + kb * BK);
                }
                // one arrival of this thread once its copies above have landed
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&bfull[stage])) : "memory");
                float* sc = sS + ring * MAX_ROWS;
                if (t < rp) sc[t] = n0;
                if (t + 64 < rp) sc[t + 64] = n1;
                if (kb + 1 < nkb) { n0 = s0[kb + 1]; n1 = s1[kb + 1]; }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sfull[ring]);
                if (++ring == stages + 2) ring = 0;
                if (++stage == stages) { stage = 0; phase ^= 1; }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // (after an abort too) copies land before the CTA leaves
    } else if (warp >= 4) {
        // ------------------------------------------ promotion and output
        const int q = warp & 3;            // TMEM lane quarter
        const int set = (warp - 4) >> 2;  // this warp's groups of 8 rows: set, set + SETS, ..
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        uint32_t slot = 0, sphase = 0;
        int ring = 0;
        uint32_t rphase = 0;
        for (int w = blockIdx.x; w < total; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = rows_pad(wk.rows);
            const int groups = (rp / 8 + SETS - 1 - set) / SETS;  // groups of 8 rows this warp promotes
            // fp8 weight scales: one per 128 x 128 block, so one per half and k block
            const int nb_per_e = p.w_rows_per_expert / MB;
            const int nb = wk.e * nb_per_e + (SWIGLU ? wk.nt : 2 * wk.nt);
            const float* ws0 = p.w_scale0 + (int64_t)nb * nkb;
            const float* ws1 = SWIGLU ? p.w_scale1 + (int64_t)nb * nkb : ws0 + nkb;
            uint64_t acc[2][4 * GROUPS];  // [half of the item][row pair]
#pragma unroll
            for (int i = 0; i < 4 * GROUPS; ++i) acc[0][i] = acc[1][i] = 0;
            float wn0 = ws0[0], wn1 = ws1[0];
            bool ok = true;
            for (int kb = 0; kb < nkb; ++kb) {
                const uint64_t wsc[2] = {pack2(wn0, wn0), pack2(wn1, wn1)};
                if (kb + 1 < nkb) { wn0 = ws0[kb + 1]; wn1 = ws1[kb + 1]; }
                const float* sc = sS + ring * MAX_ROWS;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!warp_wait(&pfull[slot], sphase, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    if (h == 0 && !warp_wait(&sfull[ring], rphase, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t t1 = t_lane + slot * SLOT_COLS + 8 * set, t2 = t1 + rp;
                    const float* f = sc + 8 * set;
                    constexpr int D = 8 * SETS;  // from one of this warp's groups to the next
#pragma unroll
                    for (int g = 0; g < GROUPS; g += 2) {  // two groups' loads in flight together
                        if (g >= groups) break;
                        uint32_t a0[8], b0[8];
                        if (g + 1 < groups) {
                            uint32_t a1[8], b1[8];
                            tmem_ld8(t1 + D * g, a0);
                            tmem_ld8(t2 + D * g, b0);
                            tmem_ld8(t1 + D * (g + 1), a1);
                            tmem_ld8(t2 + D * (g + 1), b1);
                            tmem_wait(a0, b0, a1, b1);
                            promote8(a0, b0, f + D * g, wsc[h], &acc[h][4 * g]);
                            if (g + 1 < GROUPS) promote8(a1, b1, f + D * (g + 1), wsc[h], &acc[h][4 * g + 4]);
                        } else {
                            tmem_ld8(t1 + D * g, a0);
                            tmem_ld8(t2 + D * g, b0);
                            tmem_wait(a0, b0);
                            promote8(a0, b0, f + D * g, wsc[h], &acc[h][4 * g]);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&pempty[slot]);
                    if (++slot == SLOTS) { slot = 0; sphase ^= 1; }
                }
                if (!ok) break;
                if (++ring == stages + 2) { ring = 0; rphase ^= 1; }
            }
            if (!ok) break;
            // this thread's weight row is an output column; a warp writes 64 consecutive bytes per row
            __nv_bfloat16* dst = p.out + wk.row0 * p.out_cols + wk.nt * (SWIGLU ? MB : 2 * MB) + q * 32 + lane;
#pragma unroll
            for (int i = 0; i < 4 * GROUPS; ++i) {
                const int j0 = 8 * (SETS * (i / 4) + set) + 2 * (i & 3);
                if (j0 >= wk.rows) break;
                const float2 v0 = unpack2(acc[0][i]), v1 = unpack2(acc[1][i]);
                __nv_bfloat16* o = dst + (int64_t)j0 * p.out_cols;
                if constexpr (SWIGLU) {
                    o[0] = __float2bfloat16_rn(silu_mul(v0.x, v1.x));
                    if (j0 + 1 < wk.rows) o[p.out_cols] = __float2bfloat16_rn(silu_mul(v0.y, v1.y));
                } else {
                    o[0] = __float2bfloat16_rn(v0.x);
                    o[MB] = __float2bfloat16_rn(v1.x);
                    if (j0 + 1 < wk.rows) {
                        o[p.out_cols] = __float2bfloat16_rn(v0.y);
                        o[p.out_cols + MB] = __float2bfloat16_rn(v1.y);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                     : "memory");
    }
}

// ------------------------------------------------------------------- host

template <bool SWIGLU>
static cudaError_t launch_gemm(const CUtensorMap& w0, const CUtensorMap& w1, const Params& prm, int64_t max_work,
                               cudaStream_t stream) {
    static DeviceOnce smem_set;
    const cudaError_t e = smem_set.run([] {
        return cudaFuncSetAttribute(fm_gemm_kernel<SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET);
    });
    if (e != cudaSuccess) return e;
    const int grid = (int)min64(sm_count(), max_work);
    if (grid <= 0) return cudaSuccess;
    const int stages = stages_for(prm.tile_rows);
    return launch_k(fm_gemm_kernel<SWIGLU>, dim3(grid), dim3(THREADS),
                    (size_t)FIXED_BYTES + stages * stage_bytes(prm.tile_rows), stream, w0, w1, prm, stages);
}

static bool map_e4m3(CUtensorMap* m, const void* base, int64_t rows, int64_t K) {
    return make_map(m, base, rows, K, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, BK, CU_TENSOR_MAP_SWIZZLE_128B, MB);
}

}  // namespace fm

bool ffn_fm_supported(const FfnProblem& p) {
    return p.act_dtype == GBMOE_BF16 && p.w_dtype == GBMOE_FP8_E4M3_B128 && p.H % 256 == 0 && p.I % 128 == 0 &&
           tc::encode_fn() != nullptr;
}

// Rows of a row tile: short tiles leave room for a deeper ring of weight
// stages (6 stages at 16 rows, 4 at 80)
static int fm_tile_rows(int64_t n_rows, int E) { return n_rows <= 4 * (int64_t)E ? 16 : fm::MAX_ROWS; }

cudaError_t launch_ffn_fm(const FfnProblem& p, cudaStream_t stream) {
    using namespace fm;
    if (p.n_rows == 0) return cudaSuccess;
    const int tile = fm_tile_rows(p.n_rows, p.E);
    cudaError_t err = launch_ffn_schedule(p.counts, p.E, p.n_rows, tile, p.sched, stream);
    if (err != cudaSuccess) return err;
    // every row of x once (the shared expert's rows are x's own; a routed row is a token's)
    const int64_t x_rows = p.n_rows / p.pair_div;
    if ((err = launch_quant_rows(p.x, nullptr, 1, x_rows, p.H, p.a_q, p.a_s, stream)) != cudaSuccess) return err;
    const int64_t max_m = sched_max_tiles(p.E, p.n_rows, tile);
    CUtensorMap mg, mu, md;
    if (!map_e4m3(&mg, p.w_gate, (int64_t)p.E * p.I, p.H) || !map_e4m3(&mu, p.w_up, (int64_t)p.E * p.I, p.H) ||
        !map_e4m3(&md, p.w_down, (int64_t)p.E * p.H, p.I))
        return cudaErrorInvalidValue;
    Params g{};
    g.K = p.H; g.n_tiles = p.I / MB; g.out_cols = p.I; g.w_rows_per_expert = p.I; g.tile_rows = tile;
    g.counts = p.counts; g.offsets = p.offsets; g.sched = p.sched; g.E = p.E; g.n_rows = p.n_rows;
    g.out = static_cast<__nv_bfloat16*>(p.h); g.err = p.err;
    g.q = static_cast<const uint8_t*>(p.a_q); g.plane_rows = x_rows; g.a_scale = p.a_s;
    g.gather = p.sorted_pair; g.gather_div = p.pair_div;
    g.w_scale0 = static_cast<const float*>(p.s_gate); g.w_scale1 = static_cast<const float*>(p.s_up);
    g.wait_limit_ns = tc_wait_limit_ns();
    if ((err = launch_gemm<true>(mg, mu, g, max_m * g.n_tiles, stream)) != cudaSuccess) return err;
    if ((err = launch_quant_rows(p.h, nullptr, 1, p.n_rows, p.I, p.h_q, p.h_s, stream)) != cudaSuccess) return err;
    Params d = g;
    d.K = p.I; d.n_tiles = p.H / (2 * MB); d.out_cols = p.H; d.w_rows_per_expert = p.H;
    d.out = static_cast<__nv_bfloat16*>(p.y);
    d.q = static_cast<const uint8_t*>(p.h_q); d.plane_rows = p.n_rows; d.a_scale = p.h_s;
    d.gather = nullptr; d.gather_div = 1;
    d.w_scale0 = d.w_scale1 = static_cast<const float*>(p.s_down);
    return launch_gemm<false>(md, md, d, max_m * d.n_tiles, stream);
}

}  // namespace gbmoe
