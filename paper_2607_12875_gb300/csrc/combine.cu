// Weight Sum: out[t] = sum_j w[t,j] * y_pairs[pair_pos[t*k + j]] (+ y_shared[t]).
// A thread owns 8 output columns of one token: it loads the rows of up to 8
// slots at once (a load per slot in turn left a small batch waiting out k
// latencies), then sums in slot order in fp32 and rounds once. No atomics, so
// the result does not depend on scheduling. A slot whose pair_pos is negative
// (a pair the permutation dropped) is skipped.
//
// Bound by HBM for large batches and by two dependent load latencies for small
// ones. k 8, H 4096: 32 tokens in 3.9 us (one block and a loop over the slots per
// token took 11.4), 8192 tokens in 96.8 us (98.3).
#include "common.cuh"
#include "kernels.h"

namespace gbmoe {

constexpr int kCombineThreads = 128;
constexpr int kSlots = 8;  // slots whose rows are in flight together

template <typename TA>
__global__ void __launch_bounds__(kCombineThreads)
combine_kernel(const TA* __restrict__ y, const float* __restrict__ w, const int32_t* __restrict__ pair_pos,
               const TA* __restrict__ y_shared, TA* __restrict__ out, int k, int H) {
    pdl_enter();
    const int64_t t = blockIdx.x;
    const int c = 8 * (blockIdx.y * kCombineThreads + threadIdx.x);
    if (c >= H) return;
    Raw8<TA> sh;
    if (y_shared) sh.load(y_shared + t * H + c);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int j0 = 0; j0 < k; j0 += kSlots) {
        int32_t pos[kSlots];
        float wj[kSlots];
        Raw8<TA> v[kSlots];
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            pos[j] = j0 + j < k ? pair_pos[t * k + j0 + j] : -1;
            wj[j] = j0 + j < k ? w[t * k + j0 + j] : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < kSlots; ++j)
            if (pos[j] >= 0) v[j].load(y + (int64_t)pos[j] * H + c);
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            if (pos[j] < 0) continue;  // no such slot, or a dropped pair: contributes nothing
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = __fmaf_rn(wj[j], v[j].at(i), acc[i]);
        }
    }
    if (y_shared) {
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = __fadd_rn(acc[i], sh.at(i));
    }
    Vec8<TA>::store(out + t * H + c, acc);
}

cudaError_t launch_combine(const void* y_pairs, const float* topk_w, const int32_t* pair_pos, const void* y_shared,
                           void* out, int T, int k, int H, int act_dtype, cudaStream_t stream) {
    if (T == 0) return cudaSuccess;
    const dim3 grid((unsigned)T, (unsigned)((H / 8 + kCombineThreads - 1) / kCombineThreads));
    if (act_dtype == GBMOE_BF16)
        return launch_k(combine_kernel<__nv_bfloat16>, grid, dim3(kCombineThreads), 0, stream,
                        static_cast<const __nv_bfloat16*>(y_pairs), topk_w, pair_pos,
                        static_cast<const __nv_bfloat16*>(y_shared), static_cast<__nv_bfloat16*>(out), k, H);
    return launch_k(combine_kernel<float>, grid, dim3(kCombineThreads), 0, stream, static_cast<const float*>(y_pairs), topk_w,
                    pair_pos, static_cast<const float*>(y_shared), static_cast<float*>(out), k, H);
}

}  // namespace gbmoe
