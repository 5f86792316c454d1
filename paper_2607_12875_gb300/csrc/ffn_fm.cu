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
// Activations enter as two e4m3 codes per value with one power-of-two scale s
// per row and 128 consecutive k, x = s * (q1 + 2^-kLowBits * q2): bf16's 8
// significant bits in full down to 2^-14 of the 128's largest value, and within
// 2^-22 of that value below (quant_act.cu). q2's factor 2^-kLowBits is applied in
// the promotion (short tiles) or by the MMAs, as a scale of their N operand (tall
// ones, kind::mxf8f6f4 for every format). Rows whose values spread further have
// a second pair of codes for the rest; every item then walks k twice.
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
//   1       TMEM (slots of partial sums) and the MMAs: per k block and 128-row
//           half, q1 and q2 side by side (N = 2 * rows) in short tiles, a pass
//           each into the same columns (N = rows) in tall ones;
//   2-3     gather the row codes with cp.async (the token's row of x, so no
//           sorted copy exists) and their scales;
//   4-7 or 4-11  promotion and the output: warp w reads TMEM lanes
//           32 * (w % 4).. (weight rows); in tall tiles each half of the item
//           has four warps of its own;
//   the last 4 or 8  int4: decode the tile to e4m3 codes; MXFP4: bring the weight
//           rows' scales (TMA unpacks the tile), or decode like int4 when a
//           weight pointer is not 32-byte aligned, as the unpacking TMA wants.
// A gate/up item holds 128 gate rows and the 128 up rows of the same columns, so
// gate and up of a column end up in one thread (short tiles) or in the same TMEM
// lane of two warps, which meet there once per item. Every mbarrier wait is bounded (tc_ptx.cuh).
//
// Measured, fp8, 48 tokens, top 8 of 256 experts, H 7168, I 2048 (about 2 rows
// per expert, 8.8 GB of weights): the layer 3116 -> 1302 us against the streaming
// kernels, the copy rate over its weights. What held it back on the way, per
// 128-wide k block: waits as calls (2400 -> 1750 cycles once inlined) and MMAs
// issued under `lane == 0` (1750 -> 1500).
// int4, 17 tokens, top 6 of 64 experts, H 4096, I 2816: layer 1352 -> 241 us.
// MXFP4, 16 tokens of the fp8 layer: 2893 -> 516 us. Its E8M0 scales go to the
// MMAs (kind::mxf8f6f4) and its codes are an operand as TMA unpacks them, so no
// warp touches a weight. Decoding them to e4m3 with shifts and masks was bound by
// the decode (635 us; 2.15 ms in place of 1.35 at 256 tokens), and scaling the
// codes there too, relative to the largest scale of a row's 128 k, more so (819).
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
constexpr int TMEM_COLS = 512;
constexpr int GATHER_WARPS = 2;
constexpr float kLowScale = 1.0f / (1 << kLowBits);    // of a second code
constexpr float kWideScale = 1.0f / (1 << kWideBits);  // of the second pair of planes
constexpr int SMEM_BUDGET = 232448;
// MXFP4 whose tiles TMA unpacks: 16 E2M1 codes of 8 bytes become 8 bytes and 8
// bytes of padding in shared memory, which kind::mxf8f6f4 reads as they are
// (an e2m1 operand takes as much shared memory as an e4m3 one).
constexpr int kMxfp4Unpacked = 256 + GBMOE_MXFP4;

// Per weight format and height of a row tile.
template <int WQ, int ROWS>
struct Cfg {
    // int4, MXFP4: bytes of the tile as stored, which the decode warps turn into e4m3
    static constexpr bool UNPACKED = WQ == kMxfp4Unpacked;
    static constexpr int RAW = WQ == GBMOE_FP8_E4M3_B128 || UNPACKED ? 0 : A_BYTES / 2;
    static constexpr bool BLOCK_SCALE = WQ == GBMOE_MXFP4 || UNPACKED;
    // Short tiles: a k block's two partial sums, q1 and q2 side by side, share a
    // slot of TMEM, which halves the handshakes that then dominate, and the same
    // warps promote both. Tall tiles: q1 and q2 add up in the same columns, each
    // half of the item has two slots and a set of warps of its own, and the sets
    // meet once per item (X_COL: where the up half hands its sums over).
    static constexpr bool JOINT = ROWS <= 32;
    static constexpr int SLOTS = BLOCK_SCALE && ROWS == 32 ? 3 : 4;  // (MXFP4's scales need columns too)
    static constexpr int SLOT_COLS = JOINT ? 4 * ROWS : ROWS;
    static constexpr int X_COL = SLOTS * SLOT_COLS;
    // The scale factors in TMEM of MMAs that scale. 8 columns of ones, for the
    // rows' first codes (and weights whose scales are applied in fp32); tall
    // tiles: 8 of 2^-kLowBits, for the second codes; MXFP4: weight scales, 4
    // columns per 128-row half, as many k blocks' as can have MMAs in flight: the
    // wait for a slot of partial sums then covers its scales, which the MMAs that
    // filled the slot before were the last to read.
    static constexpr bool MX = BLOCK_SCALE || !JOINT;
    static constexpr int SF_COL = X_COL + (JOINT ? 0 : ROWS);
    static constexpr int SFA_COL = SF_COL + (JOINT ? 8 : 16);
    static constexpr int SF_BLOCKS = JOINT ? SLOTS : 2;
    static constexpr int SF_COLS = MX ? SFA_COL - SF_COL + (BLOCK_SCALE ? 8 * SF_BLOCKS : 0) : 0;
    static constexpr int SF_BYTES = BLOCK_SCALE ? 2 * 512 : 0;  // a stage's weight scales in shared memory
    static constexpr int SETS = JOINT ? 1 : 2;  // of four promotion warps
    static constexpr int PROMOTE_WARPS = 4 * SETS;
    static constexpr int GROUPS = ROWS / 8;  // most groups of 8 rows
    static constexpr int HALVES_HELD = JOINT ? 2 : 1;  // halves whose sums a promotion warp holds
    static constexpr int DECODE_WARPS = RAW ? (JOINT ? 8 : 4) : 0;
    static constexpr int SCALE_WARPS = UNPACKED ? 4 : 0;
    static constexpr int THREADS = 32 * (2 + GATHER_WARPS + PROMOTE_WARPS + DECODE_WARPS + SCALE_WARPS);
    static constexpr bool SPLIT_REGS = !JOINT && DECODE_WARPS + SCALE_WARPS == 4;  // 16 warps, see setmaxnreg
    static constexpr int STAGE_BYTES = A_BYTES + RAW + SF_BYTES + 2 * ROWS * BK;
    // floats of a scale block: the rows' scales, then (int4) the weight rows'
    static constexpr int RING_FLOATS = ROWS + (WQ == GBMOE_INT4_G128 ? 2 * MB : 0);
    // UNPACKED: the ring leaves the L1 cache 60 KB. A k block reads 4 bytes of
    // scales in each of 256 lines, and eight k blocks share a sector, so the lines
    // (32 KB) have to outlive a k block: with all 228 KB as shared memory they
    // were refetched each time (sweep: 16-row tiles 597 us with 6 stages, 495 with 5 or
    // 4; 32-row tiles at 8 rows per expert 1631 with 5, 1351 with 4, 1434 with 3).
    static constexpr int MAX_STAGES = !UNPACKED ? 6 : ROWS == 16 ? 5 : ROWS == 32 ? 4 : 3;
    static constexpr int MAX_RING = MAX_STAGES + 4;
    static constexpr int NUM_BARS = 3 * MAX_STAGES + 2 * SLOTS + MAX_RING + 1 + 8;
    static constexpr int FIXED_BYTES = 1024 + MAX_RING * RING_FLOATS * 4 + NUM_BARS * 8 + 16;
    static constexpr int FIT = (SMEM_BUDGET - FIXED_BYTES) / STAGE_BYTES;
    static constexpr int STAGES = FIT < MAX_STAGES ? FIT : MAX_STAGES;
    // Scale blocks, used in turn: k block k's is written once the MMAs of
    // k - STAGES are done, which were issued once the partial sums of
    // k - STAGES - AHEAD had been promoted (TMEM holds at most AHEAD k blocks),
    // so what the block held before, k - RING's scales, has been read by then.
    static constexpr int AHEAD = JOINT ? SLOTS : 2;
    static constexpr int RING = STAGES + AHEAD;
    static constexpr int SMEM_BYTES = FIXED_BYTES + STAGES * STAGE_BYTES;
    static_assert(STAGES >= 3 && AHEAD <= 4 && SF_COL + SF_COLS <= TMEM_COLS, "ring depth");
    static_assert(ROWS % 16 == 0 && ROWS <= 128, "two rows' scales per gather thread");
};

struct Params {
    int K, n_tiles, out_cols;
    int w_rows_per_expert;  // rows of the weight tensor per expert
    int tile_rows;          // rows of a row tile of the work list
    const int32_t* counts;
    const int32_t* offsets;
    const int32_t* sched;
    int E;                   // experts of the work list (with the shared one, the last)
    int64_t n_rows;          // routed rows
    int64_t n_shared;        // rows of the shared expert, after the routed ones (0: none)
    __nv_bfloat16* out;
    int32_t* err;
    const uint8_t* q;        // code planes: [4][plane_rows][K], two pairs of q1, q2
    const int32_t* wide;     // nonzero: the second pair counts, a second walk over k multiplies it
    int64_t plane_rows;
    const float* a_scale;    // [plane_rows][K/128]
    const int32_t* gather;   // row r of the sorted order is plane row gather[r] / gather_div; null: r itself
    int gather_div;
    const void* w_scale0;    // first / second half of the item: fp8 fp32 [E, w_rows_per_expert/128, K/128],
    const void* w_scale1;    // int4 bf16 [E, w_rows_per_expert, K/128], MXFP4 E8M0 bytes [E, w_rows_per_expert, K/32]
    const void* s_scale0;    // the shared expert's
    const void* s_scale1;
    int scale_words;         // MXFP4: the E8M0 bytes are 4-byte aligned (they need only be 2-byte aligned)
    uint64_t wait_limit_ns;
};

struct Work {
    int e, nt;     // expert in its weight tensors, item of the row tile
    int64_t row0;  // first row of the tile
    int rows;      // rows in the tile
    bool shared;   // the shared expert's
};

__device__ __forceinline__ Work decode_work(const Params& p, int w) {
    const int2* tiles = reinterpret_cast<const int2*>(p.sched + sched_tiles_offset(p.E));
    const int mt = w / p.n_tiles;
    Work r;
    r.nt = w - mt * p.n_tiles;
    const int2 t = tiles[mt];
    r.shared = p.n_shared && t.x == p.E - 1;
    r.e = r.shared ? 0 : t.x;
    const int64_t cnt = r.shared ? p.n_shared : p.counts ? p.counts[t.x] : p.n_rows;
    const int64_t first = (int64_t)t.y * p.tile_rows;
    r.row0 = (r.shared ? p.n_rows : p.offsets ? p.offsets[t.x] : 0) + first;
    r.rows = (int)min64(p.tile_rows, cnt - first);
    return r;
}

// rows of one code plane in the N operand: N = 2 * rows (short tiles, both
// codes side by side) or rows (tall ones, a pass each) is a multiple of 16
template <bool SIDE>
__device__ __forceinline__ int rows_pad(int rows) { return SIDE ? (rows + 7) & ~7 : (rows + 15) & ~15; }

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

__device__ __forceinline__ void cp_async_4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// pairs of fp32, see common.cuh
__device__ __forceinline__ uint64_t pack2u(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// kind::mxf8f6f4: the same with E8M0 scales per 32 k of each operand row (bit
// 23). A k step's scale is byte j (bits 29-30 for A; B's are all ones) of the
// row's 32-bit word in TMEM.
template <bool A_E2M1>
__device__ __forceinline__ uint32_t idesc_mxf8(int n) {
    return (A_E2M1 ? 5u << 7 : 0u) | (1u << 23) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(MB >> 4) << 24);
}

__device__ __forceinline__ void mma_mxf8(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t sfa, uint32_t sfb,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb)
        : "memory");
}

// 128 rows' scale words to 4 TMEM columns: 512 bytes of shared memory, 16 per
// lane l, words 0..3 of it being rows l, 32 + l, 64 + l, 96 + l; every 32-lane
// quarter of TMEM receives them.
__device__ __forceinline__ void tmem_copy_scales(uint32_t taddr, uint32_t saddr) {
    const uint64_t desc = (uint64_t)((saddr & 0x3FFFFu) >> 4) | (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46;
    asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(desc) : "memory");
}

// 8 columns of this thread's TMEM lane, not waited for
__device__ __forceinline__ void tmem_ld8(uint32_t t, uint32_t (&a)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7])
                 : "r"(t));
}
// after the wait for the load: the registers pass through here, so that no use
// of them moves above the wait (volatile statements keep their order)
__device__ __forceinline__ void tmem_pin(uint32_t (&a)[8]) {
    asm volatile("" : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]));
}

// acc += v * (sc * w) over 8 rows: v their partial sums, sc the rows' scales in
// shared memory, w the weight scale in both halves.
__device__ __forceinline__ void promote8(const uint64_t (&v)[4], const float* sc, uint64_t w, uint64_t* acc) {
    const float4 f0 = *reinterpret_cast<const float4*>(sc), f1 = *reinterpret_cast<const float4*>(sc + 4);
    const uint64_t f[4] = {pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w)};
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = fma2(v[i], mul2(f[i], w), acc[i]);
}

// Promotes N groups of 8 rows: all their loads in flight, one wait. SIDE: the q2 sums are at t2, and added
// times 2^-kLowBits.
template <int N, bool SIDE>
__device__ __forceinline__ void promote(uint32_t t1, uint32_t t2, const float* sc, uint64_t w, uint64_t* acc) {
    uint32_t a[N][8], b[SIDE ? N : 1][8];
#pragma unroll
    for (int g = 0; g < N; ++g) {
        tmem_ld8(t1 + 8 * g, a[g]);
        if constexpr (SIDE) tmem_ld8(t2 + 8 * g, b[g]);
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int g = 0; g < N; ++g) {
        tmem_pin(a[g]);
        if constexpr (SIDE) tmem_pin(b[g]);
    }
#pragma unroll
    for (int g = 0; g < N; ++g) {
        uint64_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = pack2u(a[g][2 * i], a[g][2 * i + 1]);
            if constexpr (SIDE) v[i] = fma2(pack2u(b[g][2 * i], b[g][2 * i + 1]), pack2(kLowScale, kLowScale), v[i]);
        }
        promote8(v, sc + 8 * g, w, acc + 4 * g);
    }
}

// 8 fp32 into this thread's TMEM lane, not waited for
__device__ __forceinline__ void tmem_st8(uint32_t t, const uint64_t* v) {
    uint32_t a[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = unpack2(v[i]);
        a[2 * i] = __float_as_uint(f.x);
        a[2 * i + 1] = __float_as_uint(f.y);
    }
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(t), "r"(a[0]),
                 "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7])
                 : "memory");
}

// 16 bytes of int4 weights -> 32 e4m3 codes, the even values of each 8 before
// the odd ones. The byte m <= 8 read as e4m3 is m * 2^-9 (bits 0-2 are the
// mantissa, bit 3 the lowest exponent bit: the subnormals run on into the first
// normal binade), so the code of a nibble n is |n| with n's sign in bit 7. In
// the bytes of negative n (all ones in neg, from their sign in bit 7 of signs)
// n ^ neg is 0xf0 + |n| - 1, and 0x80 + |n| is 0x6f less. (One instruction
// decodes n + 8 for four values, but then 8 times the sum of the row's codes has
// to be taken back out in fp32, with the largest of them in it: 17 tokens of the
// layer above 219 us like that, 233 like this; 170 tokens 496 and 475.)
__device__ __forceinline__ void decode_int4_32(const uint4 raw, uint4& o0, uint4& o1) {
    auto codes = [](uint32_t signs, uint32_t w) {
        uint32_t neg;
        asm("prmt.b32 %0, %1, %1, 0xba98;" : "=r"(neg) : "r"(signs));
        return ((w & 0x0f0f0f0fu) ^ neg) - (neg & 0x6f6f6f6fu);
    };
    auto even = [&](uint32_t w) { return codes(w << 4, w); };
    auto odd = [&](uint32_t w) { return codes(w, w >> 4); };
    o0 = make_uint4(even(raw.x), odd(raw.x), even(raw.y), odd(raw.y));
    o1 = make_uint4(even(raw.z), odd(raw.z), even(raw.w), odd(raw.w));
}

// 16 bytes of MXFP4 weights -> 32 e4m3 codes in the order of int4's. The
// exponent and mantissa bits eem of an E2M1 code, put into bits 2-4 of a byte,
// read as e4m3 as the value times 2^-6 (0.5 as a subnormal too), so shifts and
// masks decode 8 values with their signs.
__device__ __forceinline__ void decode_mxfp4_32(const uint4 raw, uint4& o0, uint4& o1) {
    auto even = [](uint32_t w) { return ((w << 2) & 0x1c1c1c1cu) | ((w << 4) & 0x80808080u); };
    auto odd = [](uint32_t w) { return ((w >> 2) & 0x1c1c1c1cu) | (w & 0x80808080u); };
    o0 = make_uint4(even(raw.x), odd(raw.x), even(raw.y), odd(raw.y));
    o1 = make_uint4(even(raw.z), odd(raw.z), even(raw.w), odd(raw.w));
}

// 16-byte chunk c (0..3) of row r of a 64-byte-swizzled tile
__device__ __forceinline__ uint32_t sw64_off(int r, int c) { return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4)); }

// -------------------------------------------------------------- the GEMM

template <int WQ, int ROWS, bool SWIGLU>
__global__ void __launch_bounds__(Cfg<WQ, ROWS>::THREADS, 1)
fm_gemm_kernel(const __grid_constant__ CUtensorMap tm_w0, const __grid_constant__ CUtensorMap tm_w1,
               const __grid_constant__ CUtensorMap tm_s0, const __grid_constant__ CUtensorMap tm_s1, const Params p) {
    pdl_enter();
    using C = Cfg<WQ, ROWS>;
    constexpr int RAW = C::RAW, STAGES = C::STAGES, SLOTS = C::SLOTS, RING = C::RING;
    constexpr int B_BYTES = 2 * ROWS * BK;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sR = smem + STAGES * A_BYTES;        // int4, MXFP4: tiles as stored
    uint8_t* sB = sR + STAGES * RAW;
    uint8_t* sF = sB + STAGES * B_BYTES;          // MXFP4: weight scales
    float* sS = reinterpret_cast<float*>(sF + STAGES * C::SF_BYTES);  // [RING] scale blocks
    uint64_t* bars = reinterpret_cast<uint64_t*>(sS + RING * C::RING_FLOATS);
    uint64_t* full = bars;              // weights (decoded) and row codes of a k block are in place
    uint64_t* rfull = full + STAGES;    // int4, MXFP4: weights landed as stored
    uint64_t* empty = rfull + STAGES;   // MMAs reading the stage finished
    uint64_t* pfull = empty + STAGES;   // partial sums ready
    uint64_t* pempty = pfull + SLOTS;   // partial sums read by every promoting warp
    uint64_t* sfull = pempty + SLOTS;   // scale block written
    uint64_t* xfull = sfull + RING;     // tall tiles: the up half's sums handed over (per lane quarter)
    uint64_t* xempty = xfull + 4;       // and read
    uint64_t* drain = xempty + 4;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* walk = abort_flag + 1;  // k blocks of an item, all walks over k

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 32 * (GATHER_WARPS + C::SCALE_WARPS) + (RAW ? C::DECODE_WARPS : 1));
            mbar_init(&rfull[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < SLOTS; ++b) {
            mbar_init(&pfull[b], 1);
            mbar_init(&pempty[b], 4);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(&xfull[b], 1);
            mbar_init(&xempty[b], 1);
        }
        for (int b = 0; b < RING; ++b) mbar_init(&sfull[b], GATHER_WARPS + C::DECODE_WARPS);
        mbar_init(drain, 1);
        *abort_flag = 0;
        *walk = (*p.wide ? 2 : 1) * (p.K / BK);
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
    if constexpr (C::MX) {  // the rows' scale factors, as E8M0 bytes
        if (warp >= 4 && warp < 8) {
            const uint32_t t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + C::SF_COL;
            auto fill = [](uint32_t at, uint32_t v) {
                asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(at), "r"(v)
                             : "memory");
            };
            fill(t, 127u * 0x01010101u);
            if constexpr (!C::JOINT) fill(t + 8, (127u - kLowBits) * 0x01010101u);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }

    const int total = p.sched[1] * p.n_tiles;
    const int nkb = p.K / BK;
    const int passes = *p.wide ? 2 : 1;  // walks over k (the second: 2^-kWideBits of the first)

    // tall tiles: 16 warps start with 128 registers a thread; the promotion takes 168
    // (128 threads x (104 + 168 + 168 + 72) = 65536, what the block was launched with)
    if constexpr (C::SPLIT_REGS) {
        if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    }
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
            for (int it = 0, kb = 0; it < passes * nkb; ++it) {
                if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                inflight &= ~(1u << stage);
                constexpr int BYTES = RAW ? RAW : A_BYTES;  // (int4: 64 bytes of a row are 128 weights)
                uint8_t* dst = RAW ? sR + stage * RAW : sA + stage * A_BYTES;
                const int x = kb * (RAW ? BK / 2 : BK);
                uint64_t* bar = RAW ? &rfull[stage] : &full[stage];
                mbar_expect_tx(bar, C::UNPACKED ? BYTES / 2 : BYTES);  // (padding does not count)
                tma_load_2d(dst, wk.shared ? &tm_s0 : &tm_w0, x, a0, bar);
                tma_load_2d(dst + BYTES / 2, wk.shared ? &tm_s1 : &tm_w1, x, a1, bar);
                inflight |= 1u << stage;
                inflight_par = (inflight_par & ~(1u << stage)) | (phase << stage);
                if (++kb == nkb) kb = 0;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
        // every copy issued lands before the CTA leaves (after an abort the
        // phase may lack other arrivals: the copies get the drain limit's time)
        const uint64_t t0 = global_ns();
        for (int s = 0; s < STAGES; ++s)
            if ((inflight >> s) & 1u) drain_wait(RAW ? &rfull[s] : &full[s], (inflight_par >> s) & 1u, t0);
    } else if (warp == 1) {
        // ------------------------- MMA issuer (the whole warp, one lane issues)
        int stage = 0;
        uint32_t phase = 0;
        uint32_t kc = 0;  // k blocks so far: slot kc % SLOTS (short), 2 * half + kc % 2 (tall)
        bool ok = true, issued = false;
        const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = __shfl_sync(0xffffffffu, rows_pad<C::JOINT>(wk.rows), 0);  // warp-uniform
            const int n = C::JOINT ? 2 * rp : rp;
            const uint32_t idesc = C::MX ? idesc_mxf8<C::UNPACKED>(n) : idesc_f8(n);
            for (int it = 0; it < passes * nkb; ++it, ++kc) {
                if (!warp_wait(&full[stage], phase, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                // the row codes were written through the generic proxy (cp.async)
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                const uint64_t db = db0 + (uint64_t)(stage * B_BYTES >> 4);
                const uint64_t db2 = db + (uint64_t)(rp * BK >> 4);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint32_t slot = C::JOINT ? kc % SLOTS : 2 * half + (kc & 1);
                    const uint32_t use = C::JOINT ? kc / SLOTS : kc >> 1;
                    if (half == 0 || !C::JOINT) {
                        if (!warp_wait(&pempty[slot], (use & 1) ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                        tc_fence_after();
                    }
                    const uint32_t d = tmem_base + slot * C::SLOT_COLS + (C::JOINT ? half * 2 * ROWS : 0);
                    const uint64_t dh = da0 + (uint64_t)((stage * A_BYTES + half * (MB * BK)) >> 4);
                    const uint32_t sfb = tmem_base + C::SF_COL;
                    const uint32_t sfa = C::BLOCK_SCALE ? tmem_base + C::SFA_COL + kc % C::SF_BLOCKS * 8 + half * 4 : sfb;
                    if (elect_one()) {
                        if constexpr (C::BLOCK_SCALE)  // (a copy runs before the MMAs issued after it)
                            tmem_copy_scales(sfa, smem_u32(sF + stage * C::SF_BYTES + half * 512));
#pragma unroll
                        for (int pass = 0; pass < (C::JOINT ? 1 : 2); ++pass)
#pragma unroll
                            for (int j = 0; j < BK / 32; ++j) {  // +32 bytes along K per instruction
                                const uint32_t accumulate = pass + j != 0 ? 1u : 0u;
                                const uint64_t bj = (pass ? db2 : db) + 2 * j;
                                if constexpr (C::MX)
                                    mma_mxf8(d, dh + 2 * j, bj, idesc | (uint32_t)j << 29, sfa, sfb + 8 * pass, accumulate);
                                else mma_f8(d, dh + 2 * j, bj, idesc, accumulate);
                            }
                        if (half == 1 || !C::JOINT) mma_commit(&pfull[slot]);
                        if (half == 1) mma_commit(&empty[stage]);
                    }
                    __syncwarp();
                    issued = true;
                }
                if (!ok) break;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
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
            const int rp = rows_pad<C::JOINT>(wk.rows);
            auto src_row = [&](int j) -> int64_t {  // plane row of tile row j (past the tile's end: any valid row)
                if (j >= wk.rows) return 0;
                const int64_t r = wk.row0 + j;
                if (!p.gather) return r;
                if (wk.shared) return r - p.n_rows;
                const int32_t g = p.gather[r];
                return g >= 0 ? g / p.gather_div : 0;
            };
            const uint8_t* src[ROWS / 8];
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i) src[i] = p.q + (8 * i < rp ? src_row(r0 + 8 * i) : 0) * p.K + 16 * chunk;
            const float* s0 = p.a_scale + (t < rp ? src_row(t) : 0) * nkb;
            const float* s1 = p.a_scale + (t + 64 < rp ? src_row(t + 64) : 0) * nkb;
            for (int pass = 0; pass < passes && ok; ++pass) {
                float n0 = s0[0], n1 = s1[0];
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!warp_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    uint8_t* dst = sB + stage * B_BYTES;
#pragma unroll
                    for (int i = 0; i < ROWS / 8; ++i) {
                        if (8 * i >= rp) break;
                        const uint32_t off = sw128_off(r0 + 8 * i, chunk);
                        cp_async_16(dst + off, src[i] + kb * BK);
                        cp_async_16(dst + rp * BK + off, src[i] + plane + kb * BK);
                    }
                    // one arrival of this thread once its copies above have landed
                    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[stage])) : "memory");
                    if (pass) {  // (a block that is not finite has no second codes, and 0 times its scale would be NaN)
                        n0 = n0 < INFINITY ? n0 * kWideScale : 0.0f;
                        n1 = n1 < INFINITY ? n1 * kWideScale : 0.0f;
                    }
                    float* sc = sS + ring * C::RING_FLOATS;
                    if (t < rp) sc[t] = n0;
                    if (t + 64 < rp) sc[t + 64] = n1;
                    if (kb + 1 < nkb) { n0 = s0[kb + 1]; n1 = s1[kb + 1]; }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sfull[ring]);
                    if (++ring == RING) ring = 0;
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
#pragma unroll
                for (int i = 0; i < ROWS / 8; ++i) src[i] += 2 * plane;  // the second pair of planes
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // (after an abort too) copies land before the CTA leaves
    } else if (warp >= 4 && warp < 4 + C::PROMOTE_WARPS) {
        // ------------------------------------------ promotion and output
        if constexpr (C::SPLIT_REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 168;");
        constexpr int GROUPS = C::GROUPS;
        const int q = warp & 3;            // TMEM lane quarter
        const int set = (warp - 4) >> 2;   // tall tiles: the half of the item this warp promotes
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        uint32_t kc = 0;
        int ring = 0;
        uint32_t rphase = 0, xphase = 0;
        for (int w = blockIdx.x; w < total; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = rows_pad<C::JOINT>(wk.rows);
            const int groups = rp / 8;
            // fp8 weight scales: one per 128 x 128 block, so one per half and k block
            const int64_t nb = (int64_t)wk.e * (p.w_rows_per_expert / MB) + (SWIGLU ? wk.nt : 2 * wk.nt);
            const float* ws[2] = {static_cast<const float*>(wk.shared ? p.s_scale0 : p.w_scale0) + nb * nkb,
                                  static_cast<const float*>(wk.shared ? p.s_scale1 : p.w_scale1) + (SWIGLU ? nb : nb + 1) * nkb};
            if (!C::JOINT && set) ws[0] = ws[1];
            uint64_t acc[C::HALVES_HELD][4 * GROUPS];  // [half][row pair]
            float wn[C::HALVES_HELD];
#pragma unroll
            for (int h = 0; h < C::HALVES_HELD; ++h) {
#pragma unroll
                for (int i = 0; i < 4 * GROUPS; ++i) acc[h][i] = 0;
                wn[h] = C::UNPACKED ? 1.0f : RAW ? 64.0f : ws[h][0];  // (MXFP4's decoded codes are the values times 2^-6, the MMAs scale)
            }
            bool ok = true;
            // The count is read here: beside the accumulators there is no register to keep it in
            // (held in one, the fp8 tall tiles spill: 8192 rows of 64 experts 2.03 -> 2.15 ms).
            // MXFP4's tall tiles have one, and lose 5 % by the read (2048 tokens 2.52 -> 2.64 ms).
            for (int left = C::UNPACKED && !C::JOINT ? passes * nkb : *walk, kb = 0; left > 0; --left, ++kc) {
                if (++kb == nkb) kb = 0;  // the next block's
                float wsc[C::HALVES_HELD];
#pragma unroll
                for (int h = 0; h < C::HALVES_HELD; ++h) {
                    wsc[h] = wn[h];
                    if (!RAW && !C::UNPACKED) wn[h] = ws[h][kb];
                }
                const float* sc = sS + ring * C::RING_FLOATS;
                const uint32_t slot = C::JOINT ? kc % SLOTS : 2 * set + (kc & 1);
                const uint32_t use = C::JOINT ? kc / SLOTS : kc >> 1;
                if (!warp_wait(&sfull[ring], rphase, abort_flag, p.err, p.wait_limit_ns) ||
                    !warp_wait(&pfull[slot], use & 1, abort_flag, p.err, p.wait_limit_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < C::HALVES_HELD; ++h) {
                    // int4: one weight scale per row
                    if (WQ == GBMOE_INT4_G128) wsc[h] = sc[ROWS + (C::JOINT ? h : set) * MB + q * 32 + lane];
                    const uint64_t w2 = pack2(wsc[h], wsc[h]);
                    const uint32_t t1 = t_lane + slot * C::SLOT_COLS + h * 2 * ROWS, t2 = t1 + rp;
                    // (straight-line code per number of groups: nothing may come between loads and wait)
                    if constexpr (C::JOINT) {
#pragma unroll
                        for (int g = 0; g < GROUPS; g += 2) {
                            if (g + 1 < groups) promote<2, true>(t1 + 8 * g, t2 + 8 * g, sc + 8 * g, w2, &acc[h][4 * g]);
                            else if (g < groups) promote<1, true>(t1 + 8 * g, t2 + 8 * g, sc + 8 * g, w2, &acc[h][4 * g]);
                        }
                    } else {  // groups is even
                        static_assert(C::JOINT || GROUPS == 10);
                        if (groups >= 6) promote<6, false>(t1, 0, sc, w2, acc[h]);
                        else if (groups == 4) promote<4, false>(t1, 0, sc, w2, acc[h]);
                        else promote<2, false>(t1, 0, sc, w2, acc[h]);
                        if (groups == 8) promote<2, false>(t1 + 48, 0, sc + 48, w2, &acc[h][24]);
                        else if (groups == 10) promote<4, false>(t1 + 48, 0, sc + 48, w2, &acc[h][24]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&pempty[slot]);
                if (++ring == RING) { ring = 0; rphase ^= 1; }
            }
            if (!ok) break;
            // this thread's weight row is an output column; a warp writes 64 consecutive bytes per row
            __nv_bfloat16* dst = p.out + wk.row0 * p.out_cols + wk.nt * (SWIGLU ? MB : 2 * MB) + q * 32 + lane;
            if constexpr (C::JOINT) {
#pragma unroll
                for (int i = 0; i < 4 * GROUPS; ++i) {
                    if (2 * i >= wk.rows) break;
                    const float2 v0 = unpack2(acc[0][i]), v1 = unpack2(acc[1][i]);
                    __nv_bfloat16* o = dst + (int64_t)(2 * i) * p.out_cols;
                    if constexpr (SWIGLU) {
                        o[0] = __float2bfloat16_rn(silu_mul(v0.x, v1.x));
                        if (2 * i + 1 < wk.rows) o[p.out_cols] = __float2bfloat16_rn(silu_mul(v0.y, v1.y));
                    } else {
                        o[0] = __float2bfloat16_rn(v0.x);
                        o[MB] = __float2bfloat16_rn(v1.x);
                        if (2 * i + 1 < wk.rows) {
                            o[p.out_cols] = __float2bfloat16_rn(v0.y);
                            o[p.out_cols + MB] = __float2bfloat16_rn(v1.y);
                        }
                    }
                }
            } else if constexpr (!SWIGLU) {
#pragma unroll
                for (int i = 0; i < 4 * GROUPS; ++i) {
                    if (2 * i >= wk.rows) break;
                    const float2 v = unpack2(acc[0][i]);
                    __nv_bfloat16* o = dst + (int64_t)(2 * i) * p.out_cols + set * MB;
                    o[0] = __float2bfloat16_rn(v.x);
                    if (2 * i + 1 < wk.rows) o[p.out_cols] = __float2bfloat16_rn(v.y);
                }
            } else if (set == 1) {  // up: hand the sums to the gate half's warp of the same lanes
                if (!warp_wait(&xempty[q], xphase ^ 1, abort_flag, p.err, p.wait_limit_ns)) break;
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < GROUPS; ++g)
                    if (g < groups) tmem_st8(t_lane + C::X_COL + 8 * g, &acc[0][4 * g]);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&xfull[q]);
                xphase ^= 1;
            } else {
                if (!warp_wait(&xfull[q], xphase, abort_flag, p.err, p.wait_limit_ns)) break;
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < GROUPS; ++g) {
                    if (g >= groups) break;
                    uint32_t u[8];
                    tmem_ld8(t_lane + C::X_COL + 8 * g, u);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tmem_pin(u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int j0 = 8 * g + 2 * i;
                        const float2 v = unpack2(acc[0][4 * g + i]);
                        __nv_bfloat16* o = dst + (int64_t)j0 * p.out_cols;
                        if (j0 < wk.rows) o[0] = __float2bfloat16_rn(silu_mul(v.x, __uint_as_float(u[2 * i])));
                        if (j0 + 1 < wk.rows) o[p.out_cols] = __float2bfloat16_rn(silu_mul(v.y, __uint_as_float(u[2 * i + 1])));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&xempty[q]);
                xphase ^= 1;
            }
        }
    }
    if constexpr (C::UNPACKED) {
        if (warp >= 4 + C::PROMOTE_WARPS) {
            // ------------------------------------- weight rows' E8M0 scales
            // Thread r brings the four scales of a k block of row r of each half
            // to where the MMA issuer copies them to TMEM from.
            if constexpr (C::SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
            const int r = threadIdx.x - 32 * (4 + C::PROMOTE_WARPS);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
                const Work wk = decode_work(p, w);
                int a0, a1;
                w_rows<SWIGLU>(p, wk, a0, a1);
                const uint8_t* s0 = static_cast<const uint8_t*>(wk.shared ? p.s_scale0 : p.w_scale0) + (int64_t)(a0 + r) * nkb * 4;
                const uint8_t* s1 = static_cast<const uint8_t*>(wk.shared ? p.s_scale1 : p.w_scale1) + (int64_t)(a1 + r) * nkb * 4;
                for (int it = 0; it < passes * nkb; ++it) {
                    const int kb = it < nkb ? it : it - nkb;
                    if (!warp_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    uint8_t* dst = sF + stage * C::SF_BYTES + 16 * (r & 31) + 4 * (r >> 5);
                    if (p.scale_words) {
                        cp_async_4(dst, s0 + 4 * kb);
                        cp_async_4(dst + 512, s1 + 4 * kb);
                        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[stage])) : "memory");
                    } else {
                        const uint16_t* b0 = reinterpret_cast<const uint16_t*>(s0 + 4 * kb);
                        const uint16_t* b1 = reinterpret_cast<const uint16_t*>(s1 + 4 * kb);
                        *reinterpret_cast<uint32_t*>(dst) = b0[0] | (uint32_t)b0[1] << 16;
                        *reinterpret_cast<uint32_t*>(dst + 512) = b1[0] | (uint32_t)b1[1] << 16;
                        mbar_arrive(&full[stage]);  // (the MMA issuer has the proxy fence)
                    }
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");  // (after an abort too) copies land before the CTA leaves
        }
    }
    if constexpr (RAW) {
        if (warp >= 4 + C::PROMOTE_WARPS) {
            // ------------------------------- weight decode, weight rows' scales
            // A thread owns row r of one half (eight decode warps) or of both:
            // it decodes the row's 128 values of a k block and writes their
            // scale to the scale block (int4) or its four E8M0 scales to where
            // the MMA issuer copies them to TMEM from (MXFP4).
            if constexpr (C::SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
            constexpr int HALVES = C::DECODE_WARPS == 8 ? 1 : 2;
            const int t = threadIdx.x - 32 * (4 + C::PROMOTE_WARPS);
            const int r = t & (MB - 1), h0 = t >> 7;
            int stage = 0, ring = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
                const Work wk = decode_work(p, w);
                int a0, a1;
                w_rows<SWIGLU>(p, wk, a0, a1);
                // raw bits of the scale of k block kb of this thread's row in its half i
                auto scale_bits = [&](int i, int kb) -> uint32_t {
                    const int h = h0 + i;
                    const int64_t at = (int64_t)((h ? a1 : a0) + r) * nkb + kb;
                    const void* base = wk.shared ? (h ? p.s_scale1 : p.s_scale0) : (h ? p.w_scale1 : p.w_scale0);
                    if constexpr (WQ == GBMOE_INT4_G128) return static_cast<const uint16_t*>(base)[at];
                    if (p.scale_words) return static_cast<const uint32_t*>(base)[at];
                    const uint16_t* b = static_cast<const uint16_t*>(base) + 2 * at;
                    return b[0] | (uint32_t)b[1] << 16;
                };
                uint32_t next[HALVES];
#pragma unroll
                for (int i = 0; i < HALVES; ++i) next[i] = scale_bits(i, 0);
                for (int it = 0, kb = 0; it < passes * nkb; ++it) {
                    if (++kb == nkb) kb = 0;  // the next block's
                    uint32_t bits[HALVES];
#pragma unroll
                    for (int i = 0; i < HALVES; ++i) {
                        bits[i] = next[i];
                        next[i] = scale_bits(i, kb);
                    }
                    if (!warp_wait(&rfull[stage], phase, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                    float* sc = sS + ring * C::RING_FLOATS + ROWS;  // (int4)
#pragma unroll
                    for (int i = 0; i < HALVES; ++i) {
                        const int h = h0 + i;
                        const uint8_t* raw = sR + stage * RAW + h * (RAW / 2);
                        uint8_t* dst = sA + stage * A_BYTES + h * (A_BYTES / 2);
                        if constexpr (WQ == GBMOE_INT4_G128)
                            sc[h * MB + r] = __uint_as_float(bits[i] << 16) * 512.0f;  // bf16; the codes are n * 2^-9
                        else
                            *reinterpret_cast<uint32_t*>(sF + stage * C::SF_BYTES + h * 512 + 16 * (r & 31) + 4 * (r >> 5)) =
                                bits[i];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const uint4 v = *reinterpret_cast<const uint4*>(raw + sw64_off(r, c));
                            uint4 o0, o1;
                            if constexpr (WQ == GBMOE_INT4_G128) decode_int4_32(v, o0, o1);
                            else decode_mxfp4_32(v, o0, o1);
                            *reinterpret_cast<uint4*>(dst + sw128_off(r, 2 * c)) = o0;
                            *reinterpret_cast<uint4*>(dst + sw128_off(r, 2 * c + 1)) = o1;
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&sfull[ring]);
                        mbar_arrive(&full[stage]);
                    }
                    if (++ring == RING) ring = 0;
                    if (++stage == STAGES) { stage = 0; phase ^= 1; }
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

// ------------------------------------------------------------ bf16 weights
//
// The same item and the same way of the weights for bf16: 64 k per block, the
// rows' bf16 values as they are (one plane, gathered from x), kind::f16, and
// the sums of an item stay in tensor memory over all of K, so nothing is
// promoted: four warps read a finished slot, apply SwiGLU and store while the
// next item's MMAs fill another. 32 tokens, top 8 of 128 experts, H 4096, I
// 1536: gate/up 435 -> 405 us, down 237 -> 213 us against the streaming kernels
// (6.3 -> 6.8 TB/s).

template <int ROWS>
struct CfgBf16 {
    static constexpr int B_BYTES = ROWS * BK;  // (a block's 64 bf16 are BK bytes)
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int SLOTS = 4;
    static constexpr int SLOT_COLS = 2 * ROWS;  // both halves of an item
    static constexpr int THREADS = 32 * (2 + GATHER_WARPS + 4);
    static constexpr int MAX_STAGES = 6;
    static constexpr int FIXED_BYTES = 1024 + (2 * MAX_STAGES + 2 * SLOTS + 1) * 8 + 16;
    static constexpr int FIT = (SMEM_BUDGET - FIXED_BYTES) / STAGE_BYTES;
    static constexpr int STAGES = FIT < MAX_STAGES ? FIT : MAX_STAGES;
    static constexpr int SMEM_BYTES = FIXED_BYTES + STAGES * STAGE_BYTES;
    static_assert(SLOTS * SLOT_COLS <= TMEM_COLS && ROWS % 16 == 0, "tile");
};

// kind::f16, fp32 accumulator, bf16 x bf16, K-major, M = 128
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(MB >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

template <int ROWS, bool SWIGLU>
__global__ void __launch_bounds__(CfgBf16<ROWS>::THREADS, 1)
fm_bf16_kernel(const __grid_constant__ CUtensorMap tm_w0, const __grid_constant__ CUtensorMap tm_w1, const Params p) {
    pdl_enter();
    using C = CfgBf16<ROWS>;
    constexpr int STAGES = C::STAGES, SLOTS = C::SLOTS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * A_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(sB + STAGES * C::B_BYTES);  // weights and rows of a k block landed
    uint64_t* empty = full + STAGES;                                         // MMAs reading the stage finished
    uint64_t* pfull = empty + STAGES;                                        // an item's sums are complete
    uint64_t* pempty = pfull + SLOTS;                                        // and read by every epilogue warp
    uint64_t* drain = pempty + SLOTS;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 32 * GATHER_WARPS + 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < SLOTS; ++b) {
            mbar_init(&pfull[b], 1);
            mbar_init(&pempty[b], 4);
        }
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
    const int nkb = p.K / (BK / 2);
    auto pad16 = [](int rows) { return (rows + 15) & ~15; };

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
                uint8_t* dst = sA + stage * A_BYTES;
                mbar_expect_tx(&full[stage], A_BYTES);
                tma_load_2d(dst, &tm_w0, kb * (BK / 2), a0, &full[stage]);
                tma_load_2d(dst + A_BYTES / 2, &tm_w1, kb * (BK / 2), a1, &full[stage]);
                inflight |= 1u << stage;
                inflight_par = (inflight_par & ~(1u << stage)) | (phase << stage);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
        // every copy issued lands before the CTA leaves (after an abort the
        // phase may lack other arrivals: the copies get the drain limit's time)
        const uint64_t t0 = global_ns();
        for (int s = 0; s < STAGES; ++s)
            if ((inflight >> s) & 1u) drain_wait(&full[s], (inflight_par >> s) & 1u, t0);
    } else if (warp == 1) {
        // ------------------------- MMA issuer (the whole warp, one lane issues)
        int stage = 0;
        uint32_t phase = 0;
        uint32_t slot = 0, sphase = 0;
        bool ok = true, issued = false;
        const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const uint32_t idesc = idesc_bf16(__shfl_sync(0xffffffffu, pad16(wk.rows), 0));  // warp-uniform
            if (!warp_wait(&pempty[slot], sphase ^ 1, abort_flag, p.err, p.wait_limit_ns)) break;
            tc_fence_after();
            const uint32_t d = tmem_base + slot * C::SLOT_COLS;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!warp_wait(&full[stage], phase, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                // the rows were written through the generic proxy (cp.async)
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                const uint64_t db = db0 + (uint64_t)(stage * C::B_BYTES >> 4);
                const uint64_t da = da0 + (uint64_t)(stage * A_BYTES >> 4);
                if (elect_one()) {
#pragma unroll
                    for (int half = 0; half < 2; ++half)
#pragma unroll
                        for (int j = 0; j < BK / 32; ++j)  // 16 k, +32 bytes, per instruction
                            mma_bf16(d + half * ROWS, da + (uint64_t)(half * (MB * BK) >> 4) + 2 * j, db + 2 * j, idesc,
                                     (kb | j) != 0 ? 1u : 0u);
                    mma_commit(&empty[stage]);
                    if (kb == nkb - 1) mma_commit(&pfull[slot]);
                }
                __syncwarp();
                issued = true;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            if (++slot == SLOTS) { slot = 0; sphase ^= 1; }
        }
        if (issued) {  // every MMA issued has finished before TMEM is released
            if (elect_one()) mma_commit(drain);
            __syncwarp();
            drain_wait(drain, 0);
        }
    } else if (warp >= 2 && warp < 2 + GATHER_WARPS) {
        // --------------------------------------------------- row gather
        // thread t copies 16-byte chunk t % 8 of rows t / 8 + 8 i
        const int t = threadIdx.x - 64;
        const int chunk = t & 7, r0 = t >> 3;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            const int rp = pad16(wk.rows);
            const uint8_t* src[ROWS / 8];
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i) {  // (rows past the tile's end: any valid row, never stored)
                const int j = r0 + 8 * i;
                int64_t row = 0;
                if (j < wk.rows) {
                    row = wk.row0 + j;
                    if (p.gather) {
                        const int32_t g = p.gather[row];
                        row = g >= 0 ? g / p.gather_div : 0;
                    }
                }
                src[i] = p.q + row * p.K * 2 + 16 * chunk;
            }
            for (int kb = 0; kb < nkb; ++kb) {
                if (!warp_wait(&empty[stage], phase ^ 1, abort_flag, p.err, p.wait_limit_ns)) { ok = false; break; }
                uint8_t* dst = sB + stage * C::B_BYTES;
#pragma unroll
                for (int i = 0; i < ROWS / 8; ++i) {
                    if (8 * i >= rp) break;
                    cp_async_16(dst + sw128_off(r0 + 8 * i, chunk), src[i] + kb * BK);
                }
                // one arrival of this thread once its copies above have landed
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&full[stage])) : "memory");
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // (after an abort too) copies land before the CTA leaves
    } else if (warp >= 4) {
        // -------------------------------------------------------- epilogue
        const int q = warp & 3;  // TMEM lane quarter
        const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
        uint32_t slot = 0, sphase = 0;
        for (int w = blockIdx.x; w < total; w += gridDim.x) {
            const Work wk = decode_work(p, w);
            if (!warp_wait(&pfull[slot], sphase, abort_flag, p.err, p.wait_limit_ns)) break;
            tc_fence_after();
            // this thread's weight row is an output column; a warp writes 64 consecutive bytes per row
            __nv_bfloat16* dst = p.out + wk.row0 * p.out_cols + wk.nt * (SWIGLU ? MB : 2 * MB) + q * 32 + lane;
            const uint32_t t1 = t_lane + slot * C::SLOT_COLS;
            for (int j0 = 0; j0 < wk.rows; j0 += 8) {
                uint32_t a[8], b[8];
                tmem_ld8(t1 + j0, a);
                tmem_ld8(t1 + ROWS + j0, b);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                tmem_pin(a);
                tmem_pin(b);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (j0 + i >= wk.rows) break;
                    __nv_bfloat16* o = dst + (int64_t)(j0 + i) * p.out_cols;
                    const float v0 = __uint_as_float(a[i]), v1 = __uint_as_float(b[i]);
                    if constexpr (SWIGLU) {
                        o[0] = __float2bfloat16_rn(silu_mul(v0, v1));
                    } else {
                        o[0] = __float2bfloat16_rn(v0);
                        o[MB] = __float2bfloat16_rn(v1);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&pempty[slot]);
            if (++slot == SLOTS) { slot = 0; sphase ^= 1; }
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

template <int WQ, int ROWS, bool SWIGLU>
static cudaError_t launch_gemm(const CUtensorMap& w0, const CUtensorMap& w1, const CUtensorMap& s0,
                               const CUtensorMap& s1, const Params& prm, int64_t max_work, cudaStream_t stream) {
    using C = Cfg<WQ, ROWS>;
    static DeviceOnce smem_set;
    const cudaError_t e = smem_set.run([] {
        return cudaFuncSetAttribute(fm_gemm_kernel<WQ, ROWS, SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    C::SMEM_BYTES);
    });
    if (e != cudaSuccess) return e;
    const int grid = (int)min64(sm_count(), max_work);
    if (grid <= 0) return cudaSuccess;
    return launch_k(fm_gemm_kernel<WQ, ROWS, SWIGLU>, dim3(grid), dim3(C::THREADS), C::SMEM_BYTES, stream, w0, w1, s0, s1,
                    prm);
}

// [rows, K] weights in boxes of 128 rows x 128 k as stored
static bool map_weights(CUtensorMap* m, int wq, const void* base, int64_t rows, int64_t K) {
    if (wq == kMxfp4Unpacked) {
        // wants a 32-byte aligned base, strides that are multiples of 32 bytes,
        // extents of multiples of 128 codes and boxes of 128 codes
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
        const cuuint64_t strides[1] = {(cuuint64_t)K / 2};
        const cuuint32_t box[2] = {BK, MB};
        const cuuint32_t estr[2] = {1, 1};
        return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_16U4_ALIGN16B, 2, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    if (wq != GBMOE_FP8_E4M3_B128)
        return make_map(m, base, rows, K / 2, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, BK / 2, CU_TENSOR_MAP_SWIZZLE_64B, MB);
    return make_map(m, base, rows, K, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, BK, CU_TENSOR_MAP_SWIZZLE_128B, MB);
}

template <int WQ, int ROWS>
static cudaError_t launch_ffn(const FfnProblem& p, cudaStream_t stream) {
    const int tile = ROWS;
    cudaError_t err = launch_ffn_schedule(p.counts, p.E, p.n_rows, tile, p.sched, stream, p.n_shared);
    if (err != cudaSuccess) return err;
    const int experts = p.E + (p.n_shared ? 1 : 0);
    const int64_t rows = p.n_rows + p.n_shared;
    // every row of x once (the shared expert's rows are x's own; a routed row is a token's)
    const int64_t x_rows = p.n_rows / p.pair_div;
    constexpr bool kFour = Cfg<WQ, ROWS>::RAW != 0;  // the order 4-bit weights are decoded in
    if ((err = launch_quant_planes(p.x, x_rows, p.H, p.a_q, p.a_s, kFour, p.sched + kSchedWideX, nullptr, 0, stream)) != cudaSuccess)
        return err;
    const int64_t max_m = sched_max_tiles(experts, rows, tile);
    CUtensorMap mg, mu, md, sg, su, sd;
    if (!map_weights(&mg, WQ, p.w_gate, (int64_t)p.E * p.I, p.H) ||
        !map_weights(&mu, WQ, p.w_up, (int64_t)p.E * p.I, p.H) ||
        !map_weights(&md, WQ, p.w_down, (int64_t)p.E * p.H, p.I))
        return cudaErrorInvalidValue;
    sg = mg; su = mu; sd = md;
    if (p.n_shared && (!map_weights(&sg, WQ, p.sw_gate, p.I, p.H) || !map_weights(&su, WQ, p.sw_up, p.I, p.H) ||
                       !map_weights(&sd, WQ, p.sw_down, p.H, p.I)))
        return cudaErrorInvalidValue;
    Params g{};
    g.K = p.H; g.n_tiles = p.I / MB; g.out_cols = p.I; g.w_rows_per_expert = p.I; g.tile_rows = tile;
    g.counts = p.counts; g.offsets = p.offsets; g.sched = p.sched; g.E = experts; g.n_rows = p.n_rows;
    g.n_shared = p.n_shared;
    g.out = static_cast<__nv_bfloat16*>(p.h); g.err = p.err;
    g.q = static_cast<const uint8_t*>(p.a_q); g.plane_rows = x_rows; g.a_scale = p.a_s; g.wide = p.sched + kSchedWideX;
    g.gather = p.sorted_pair; g.gather_div = p.pair_div;
    g.w_scale0 = p.s_gate; g.w_scale1 = p.s_up; g.s_scale0 = p.ss_gate; g.s_scale1 = p.ss_up;
    auto words = [](const void* s) { return reinterpret_cast<uintptr_t>(s) % 4 == 0; };
    g.scale_words = words(p.s_gate) && words(p.s_up) && words(p.ss_gate) && words(p.ss_up);
    g.wait_limit_ns = tc_wait_limit_ns();
    if ((err = launch_gemm<WQ, ROWS, true>(mg, mu, sg, su, g, max_m * g.n_tiles, stream)) != cudaSuccess) return err;
    // (rows of h past the last kept pair were not written)
    if ((err = launch_quant_planes(p.h, rows, p.I, p.h_q, p.h_s, kFour, p.sched + kSchedWideH, p.offsets ? p.offsets + p.E : nullptr,
                                   p.offsets ? p.n_rows : 0, stream)) != cudaSuccess)
        return err;
    Params d = g;
    d.K = p.I; d.n_tiles = p.H / (2 * MB); d.out_cols = p.H; d.w_rows_per_expert = p.H;
    d.out = static_cast<__nv_bfloat16*>(p.y);
    d.q = static_cast<const uint8_t*>(p.h_q); d.plane_rows = rows; d.a_scale = p.h_s; d.wide = p.sched + kSchedWideH;
    d.gather = nullptr; d.gather_div = 1;
    d.w_scale0 = d.w_scale1 = p.s_down; d.s_scale0 = d.s_scale1 = p.ss_down;
    d.scale_words = words(p.s_down) && words(p.ss_down);
    return launch_gemm<WQ, ROWS, false>(md, md, sd, sd, d, max_m * d.n_tiles, stream);
}

// Rows of a row tile: short ones leave shared memory for more weight stages
// (fp8: 6 at 16 rows, 5 at 32, 4 at 80) and warps for the decode (eight, not
// four), and pass both partial sums of a k block at once; an expert with more
// rows takes several tiles, whose weights come from L2. MXFP4, 256 experts,
// H 7168, I 2048: 2.82 -> 2.15 ms at 8 rows per expert with 32-row tiles in
// place of 80-row ones, 2.90 -> 2.26 at 16; fp8 1.83 -> 1.81 and 1.90 -> 1.88.
constexpr int64_t kShortRowsPerExpert = 16;

template <int WQ>
static cudaError_t launch_ffn(const FfnProblem& p, cudaStream_t stream) {
    if (p.n_rows <= 4 * (int64_t)p.E) return launch_ffn<WQ, 16>(p, stream);
    return p.n_rows <= kShortRowsPerExpert * p.E ? launch_ffn<WQ, 32>(p, stream) : launch_ffn<WQ, 80>(p, stream);
}

template <int ROWS, bool SWIGLU>
static cudaError_t launch_gemm_bf16(const CUtensorMap& w0, const CUtensorMap& w1, const Params& prm, int64_t max_work,
                                    cudaStream_t stream) {
    using C = CfgBf16<ROWS>;
    static DeviceOnce smem_set;
    const cudaError_t e = smem_set.run([] {
        return cudaFuncSetAttribute(fm_bf16_kernel<ROWS, SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    });
    if (e != cudaSuccess) return e;
    const int grid = (int)min64(sm_count(), max_work);
    if (grid <= 0) return cudaSuccess;
    return launch_k(fm_bf16_kernel<ROWS, SWIGLU>, dim3(grid), dim3(C::THREADS), C::SMEM_BYTES, stream, w0, w1, prm);
}

template <int ROWS>
static cudaError_t launch_ffn_bf16(const FfnProblem& p, cudaStream_t stream) {
    cudaError_t err = launch_ffn_schedule(p.counts, p.E, p.n_rows, ROWS, p.sched, stream);
    if (err != cudaSuccess) return err;
    const int64_t max_m = sched_max_tiles(p.E, p.n_rows, ROWS);
    auto map = [](CUtensorMap* m, const void* base, int64_t rows, int64_t K) {
        return make_map(m, base, rows, K * 2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, BK / 2, CU_TENSOR_MAP_SWIZZLE_128B, MB);
    };
    CUtensorMap mg, mu, md;
    if (!map(&mg, p.w_gate, (int64_t)p.E * p.I, p.H) || !map(&mu, p.w_up, (int64_t)p.E * p.I, p.H) ||
        !map(&md, p.w_down, (int64_t)p.E * p.H, p.I))
        return cudaErrorInvalidValue;
    Params g{};
    g.K = p.H; g.n_tiles = p.I / MB; g.out_cols = p.I; g.w_rows_per_expert = p.I; g.tile_rows = ROWS;
    g.counts = p.counts; g.offsets = p.offsets; g.sched = p.sched; g.E = p.E; g.n_rows = p.n_rows;
    g.out = static_cast<__nv_bfloat16*>(p.h); g.err = p.err;
    g.q = static_cast<const uint8_t*>(p.x);
    g.gather = p.sorted_pair; g.gather_div = p.pair_div;
    g.wait_limit_ns = tc_wait_limit_ns();
    if ((err = launch_gemm_bf16<ROWS, true>(mg, mu, g, max_m * g.n_tiles, stream)) != cudaSuccess) return err;
    Params d = g;
    d.K = p.I; d.n_tiles = p.H / (2 * MB); d.out_cols = p.H; d.w_rows_per_expert = p.H;
    d.out = static_cast<__nv_bfloat16*>(p.y);
    d.q = static_cast<const uint8_t*>(p.h);
    d.gather = nullptr; d.gather_div = 1;
    return launch_gemm_bf16<ROWS, false>(md, md, d, max_m * d.n_tiles, stream);
}

}  // namespace fm

bool ffn_fm_supported(const FfnProblem& p) {
    const bool wq_ok = p.w_dtype == GBMOE_BF16 || p.w_dtype == GBMOE_FP8_E4M3_B128 || p.w_dtype == GBMOE_INT4_G128 || p.w_dtype == GBMOE_MXFP4;
    return p.act_dtype == GBMOE_BF16 && wq_ok && p.H % 256 == 0 && p.I % 128 == 0 && tc::encode_fn() != nullptr;
}

cudaError_t launch_ffn_fm(const FfnProblem& p, cudaStream_t stream) {
    if (p.n_rows == 0) return cudaSuccess;
    switch (p.w_dtype) {
        case GBMOE_BF16:
            return p.n_rows <= 4 * (int64_t)p.E ? fm::launch_ffn_bf16<16>(p, stream) : fm::launch_ffn_bf16<64>(p, stream);
        case GBMOE_FP8_E4M3_B128: return fm::launch_ffn<GBMOE_FP8_E4M3_B128>(p, stream);
        case GBMOE_INT4_G128: return fm::launch_ffn<GBMOE_INT4_G128>(p, stream);
        case GBMOE_MXFP4: {
            auto aligned = [](const void* w) { return reinterpret_cast<uintptr_t>(w) % 32 == 0; };  // (or null: no shared expert)
            const bool unpacked = aligned(p.w_gate) && aligned(p.w_up) && aligned(p.w_down) && aligned(p.sw_gate) &&
                                  aligned(p.sw_up) && aligned(p.sw_down);
            return unpacked ? fm::launch_ffn<fm::kMxfp4Unpacked>(p, stream) : fm::launch_ffn<GBMOE_MXFP4>(p, stream);
        }
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace gbmoe
