// Internal launch interface between the C ABI (api.cu) and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gbmoe.h"

namespace gbmoe {

struct RouteParams {
    int T, H, E, top_k;
    int score, renormalize, n_group, topk_group;
    float routed_scale;
    int act_dtype;
    int gate_tc;  // 1: logits on the tensor cores, audited against the fixed order
};

// scratch of the tensor-core gate: schedule ints for T rows, the device error
// word, two words for the audit (max router row norm, count of flagged
// tokens) and the list of flagged tokens [T]
struct RouteScratch {
    int32_t* sched;
    int32_t* err;
    float* audit;
    int32_t* flagged;
};

// logits: fp32 scratch, T * E floats (gate_tc: gate_tc_splits planes of them); topk_ids, topk_w [T, k]
cudaError_t launch_route(const RouteParams& rp, const void* x, const void* w_router, const float* logit_bias,
                         const float* select_bias, float* logits, int32_t* topk_ids, float* topk_w,
                         const RouteScratch& rs, cudaStream_t stream);
// RMSNorm of x [T, H] (act dtype) with gamma [H] into y, in the gate's order
cudaError_t launch_rmsnorm(const void* x, const void* gamma, float eps, int T, int H, int act_dtype, void* y,
                           cudaStream_t stream);
// router logits on the tensor cores (bf16 x and router weight; ffn_tc.cu), as
// gate_tc_splits partial planes [splits, T, E] without the bias
int gate_tc_splits(int T, int H, int E);
cudaError_t launch_gate_tc(const void* x, const void* wg, float* logits, int T, int H, int E, int32_t* sched,
                           int32_t* err, cudaStream_t stream);

// Number of 1024-pair blocks the permutation uses, and its scratch ints.
int permute_blocks(int64_t P);
size_t permute_scratch_ints(int64_t P, int E);
cudaError_t launch_permute(const int32_t* topk_ids, int64_t P, int E, int32_t* counts, int32_t* offsets,
                           int32_t* sorted_pair, int32_t* pair_pos, int32_t* scratch, cudaStream_t stream);

// One grouped FFN problem: rows r of expert e are offsets[e] .. offsets[e+1]-1,
// the token of row r is sorted_pair[r] / pair_div (r itself when sorted_pair
// is null). counts null means one expert with n_rows rows.
struct FfnProblem {
    const void* x;              // [T, H] act
    const int32_t* counts;      // [E] or null
    const int32_t* offsets;     // [E+1] or null (then 0, n_rows)
    const int32_t* sorted_pair; // [rows] or null
    const int32_t* pair_pos;    // its inverse [rows], or null when the caller does not have it
    int pair_div;
    int E, H, I;
    int64_t n_rows;             // upper bound on rows (P, or T for the shared expert)
    int act_dtype, w_dtype;
    const void *w_gate, *w_up, *w_down, *s_gate, *s_up, *s_down;
    void* y;                    // [n_rows, H] act
    // scratch carved by the caller
    void* h;                    // [n_rows, I] act
    void* x_sorted;             // [n_rows, H] act: the sorted copy the quantised-weight one-CTA GEMM and the
                                // CTA-pair GEMMs read (null on routes that do not use one)
    void* w_dq;                 // bf16 [E, I, H] gate, [E, I, H] up, [E, H, I] down, or null:
                                // quantised weights are then decoded once into it (TC_DEQUANT)
    void* a_q;                  // routes that multiply e4m3 codes: x as two e4m3 code planes (value and
                                //   residual), [2, rows, H] in sorted order (row-major fp8 GEMM) or two
                                //   pairs, [4, T, H] in token order (feature-major GEMM)
    float* a_s;                 //   and their 1x128 scales [rows, H/128]
    void* h_q;                  //   h the same way, [2 or 4, n_rows, I]
    float* h_s;                 //   and its 1x128 scales [n_rows, I/128]
    // Feature-major GEMM: the shared expert (same I and weight format) as one more
    // expert of the problem, its n_shared rows (token order) after the routed
    // ones in h, y and h's codes; 0: none
    int64_t n_shared;
    const void *sw_gate, *sw_up, *sw_down, *ss_gate, *ss_up, *ss_down;
    int cta_pair;               // tensor-core routes: 1 = CTA pairs (cta_group::2, 256-row M tiles)
    int32_t* sched;             // schedule ints, ffn_sched_ints(E, n_rows)
    int32_t* err;               // device error word
    // Weight Sum fused into the down GEMM (tensor-core routes; fuse_k = top_k,
    // 0 = off): y then receives topk_w[p] * y of pair p at row p (pair order)
    // and out_final[t] = sum_j slots of t (+ y_shared[t]); arrive holds
    // T * (H / 256) zeroed counters
    int fuse_k;
    const float* topk_w;
    const void* y_shared;
    void* out_final;
    int32_t* arrive;
};

size_t ffn_sched_ints(int E, int64_t n_rows);
// AUTO: 4-bit weights are decoded once (TC_DEQUANT) from this many rows per
// expert on; below, inside the GEMM. With few weights in all the decode pass costs
// little and its bf16 copy stays in L2; with many it is a full round trip through
// HBM, while the GEMM has work items enough to hide its own decode. In the GEMM
// against decoded once, us: 24 experts, H 1024, I 512 (13 M weights a matrix) 114
// and 103 at 256 rows per expert; 24, 2048, 1024 (50 M) 222 and 221 at 260; 48, 3072,
// 1024 (151 M) 478 and 498 at 260, 534 and 526 at 300; 40, 4096, 1408 (231 M) 724 and
// 746 at 349, 910 and 842 at 399; 64, 4096, 2816 (738 M) 2018 and 2184 at 349, 2432 and
// 2428 at 399. (278, 5632, 128: layer 1570 and 1431 at 317.)
inline int64_t dequant_rows_per_expert(int E, int H, int I) {
    const int64_t weights = (int64_t)E * H * I;
    return weights < 90000000 ? 256 : weights < 200000000 || I < 512 ? 288 : weights < 400000000 ? 352 : 384;
}
// AUTO: CTA pairs from this many rows per expert on. bf16, 128 experts, H 4096,
// I 1536, pairs against single CTAs: 2.245 and 2.252 ms at 512 rows per expert,
// 3.93 and 3.99 at 1024.
constexpr int64_t kPairRowsPerExpert = 1024;
// After a decode-once pass, with wide experts and enough 256-row items, from here
// on (pairs against single CTAs, us: I 4096, 8 experts, H 4096, 486 and 546 at 400
// rows per expert; I 2816 2488 and 2627 at 499; I 1280, 16 experts, H 4096, 359 and 352
// at 400, 440 and 458 at 700; I 512, 40 experts, 560 and 512 at 700; one expert of I
// 2688, H 1536, 809 rows: layer 106 and 101).
constexpr int64_t kPairDequantRowsPerExpert = 400;
constexpr int kPairDequantMinWidth = 1280;  // H and I
constexpr int64_t kPairDequantMinItems = 256;  // of 256 rows x 128 gate and up rows
// bf16 weights stream on the CUDA cores below this many rows per expert: a
// weight then meets one row or two, and the streaming CTAs split a few experts'
// weights finer than the feature-major items (the same layer at 0.06 rows per
// expert: 71 us streaming against 73, 0.13: 111 against 120, 0.5: 299 against
// 306).
constexpr int64_t kFmBf16MinRowsPerExpert = 1;
// A layer with few rows in all streams, in any format: up to 1 + few_rows * (1/H +
// 1/I) rows. Streaming splits an expert's weights over the SMs, and its time grows with
// rows x H x I; the feature-major GEMM with few items on its list (I / 128 per
// expert with rows, H / 256 in the down GEMM) takes H / 128 and then I / 128 k
// blocks one after the other, whatever the rows. Where the two meet was measured
// on 14 shapes from H 1024, I 768 to H 4096, I 6144 and from 1 expert to 128,
// 1 to 96 rows: the lines below are within 11 % of the better one everywhere, and on
// the streaming side where it is close. Streaming against feature-major, one expert, H 4096, I 1536, with
// the gate: bf16 31 against 51 us at 1 row, 49 against 53 at 6, 57 against 55 at 16;
// fp8 29 and 46 at 1, 53 and 48 at 6; int4 30 and 56 at 1, 63 and 59 at 6; MXFP4 36
// and 50 at 1, 53 and 51 at 3. 8 experts, top 2, H 2048, I 512: fp8 26 and 34 at 2
// rows, 38 and 36 at 16.
constexpr double few_rows(int w_dtype) {
    return w_dtype == GBMOE_BF16            ? 12000.0
           : w_dtype == GBMOE_FP8_E4M3_B128 ? 5000.0
           : w_dtype == GBMOE_INT4_G128     ? 4800.0
           : w_dtype == GBMOE_MXFP4         ? 1600.0
                                            : 0.0;
}
cudaError_t launch_ffn_stream(const FfnProblem& p, cudaStream_t stream);
size_t stream_smem_bytes(int act_dtype, int H, int I);  // per CTA, streaming route
// dynamic shared memory a CTA may use on sm_103a (227 KB); a streaming problem
// runs when its stream_smem_bytes fits
constexpr size_t stream_smem_budget() { return 227 * 1024; }
cudaError_t launch_ffn_simt(const FfnProblem& p, cudaStream_t stream);
cudaError_t launch_ffn_tc(const FfnProblem& p, cudaStream_t stream);
bool ffn_tc_supported(const FfnProblem& p);
bool ffn_tc_pair_supported(const FfnProblem& p);
cudaError_t launch_ffn_tc_fp8(const FfnProblem& p, cudaStream_t stream);
bool ffn_tc_fp8_supported(const FfnProblem& p);
// The feature-major GEMM runs up to this many rows per expert; beyond, the
// 128-row MMAs of the row-major GEMMs waste less than its second pass over the
// weights' operand costs. Feature-major against row-major, 256 experts, H 7168,
// I 2048: fp8 2.14 against 2.48 ms at 32 rows per expert, 2.37 against 2.52 at
// 47, 2.83 against 2.66 at 64; MXFP4 2.56 against 3.43 (decode in the GEMM) at
// 32, 2.81 against 3.39 at 47, 3.23 against 3.47 at 64, 3.65 against 3.55 at 72 (with decode warps, at
// unaligned weights, 3.46 at 64); int4, 64 experts, H 4096, I 2816: 0.59 against
// 0.78 at 24, 0.78 against 0.78 at 48, 0.96 against 0.85 at 72; bf16, 128 experts, H 4096, I 1536: 0.775
// against 0.800 at 21, 0.62 against 0.70 (streaming) at 2.
// fp8 with narrow inputs leaves the gate/up items two or four k blocks, less than
// their handover of sums costs: 128 experts, I 3072, H 256 1.07 times the speed of
// the row-major GEMM (before its stacked tiles) at 28 rows, 0.97 at 36, 0.85 at 52; H
// 512 1.00 at 44, 0.95 at 52; H 1024 1.02 at 52.
inline int64_t fm_fp8_rows_per_expert(int H) { return H >= 1024 ? 52 : H >= 512 ? 40 : 28; }
constexpr int64_t kFmMxfp4RowsPerExpert = 64;
constexpr int64_t kFmRowsPerExpert = 40;
// The feature-major GEMM's activation codes (quant_act.cu): factor 2^-kLowBits between the second codes and the
// first, and 2^-kWideBits between the second pair of planes and the first.
constexpr int kLowBits = 5, kWideBits = 22;
// Rows of src (bf16) as four e4m3 code planes [4, n_rows, K] and 1x128 scales [n_rows, K / 128]; *wide is set when
// the second pair counts. four_bit: in the order 4-bit weights are decoded in. With kept, rows *kept .. n_routed - 1
// are left out (positions of dropped pairs).
cudaError_t launch_quant_planes(const void* src, int64_t n_rows, int K, void* q, float* s, bool four_bit, int32_t* wide,
                                const int32_t* kept, int64_t n_routed, cudaStream_t stream);
// rows of src (gathered when gather is set) as the row-major GEMM's two code planes [2, n_rows, K], and scales
cudaError_t launch_quant_rows(const void* src, const int32_t* gather, int gather_div, int64_t n_rows, int K, void* q,
                              float* s, cudaStream_t stream);
// the same of every row of src once, row r's codes written to rows pair_pos[r * k ..] of [2, n_src * k, K]
cudaError_t launch_quant_scatter(const void* src, const int32_t* pair_pos, int k, int64_t n_src, int K, void* q, float* s,
                                 cudaStream_t stream);
cudaError_t launch_ffn_fm(const FfnProblem& p, cudaStream_t stream);
bool ffn_fm_supported(const FfnProblem& p);

cudaError_t launch_combine(const void* y_pairs, const float* topk_w, const int32_t* pair_pos, const void* y_shared,
                           void* out, int T, int k, int H, int act_dtype, cudaStream_t stream);

}  // namespace gbmoe
