// Weight Sum: out[t] = sum_j w[t,j] * y_pairs[pair_pos[t*k + j]] (+ y_shared[t]).
// A thread owns 8 output columns of one token at a time: it loads the rows of up
// to 8 slots at once (a load per slot in turn left a small batch waiting out k
// latencies), then sums in slot order in fp32 and rounds once. No atomics, so the
// result does not depend on scheduling. A slot whose pair_pos is negative (a pair
// the permutation dropped) is skipped.
//
// Bound by HBM for large batches and by two dependent load latencies for small
// ones. A batch takes a block per token and 128 threads' columns as far as that
// fills the SMs, beyond it a block walks its token's row and reads the slots once;
// the slots in flight go with k, to 4 for fp32 rows (8 take half the threads).
// bf16, H 4096, us: 64 tokens of k 8 1.8 (one block per token, a loop over its slots
// 4.5); 16384 of k 1 42.3 (8 slots for every k and a thread per 8 columns 101, the
// block and loop 47), of k 8 174 (190, 193).
#include "common.cuh"
#include "kernels.h"

namespace gbmoe {

constexpr int kCombineThreads = 128;
constexpr int kBlocksPerSm = 16;  // resident at once

// kSlots: slots whose rows are in flight together
template <typename TA, int kSlots>
__global__ void __launch_bounds__(kCombineThreads)
combine_kernel(const TA* __restrict__ y, const float* __restrict__ w, const int32_t* __restrict__ pair_pos,
               const TA* __restrict__ y_shared, TA* __restrict__ out, int k, int H) {
    pdl_enter();
    const int64_t t = blockIdx.x;
    int32_t pos[kSlots];
    float wj[kSlots];
    auto slots = [&](int j0) {  // no such slot: as one of a dropped pair
#pragma unroll
        for (int j = 0; j < kSlots; ++j) {
            pos[j] = j0 + j < k ? pair_pos[t * k + j0 + j] : -1;
            wj[j] = j0 + j < k ? w[t * k + j0 + j] : 0.0f;
        }
    };
    slots(0);
    for (int c = 8 * (blockIdx.y * kCombineThreads + threadIdx.x); c < H; c += 8 * kCombineThreads * gridDim.y) {
        Raw8<TA> sh;
        if (y_shared) sh.load(y_shared + t * H + c);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int j0 = 0; j0 < k; j0 += kSlots) {
            if (k > kSlots) slots(j0);
            Raw8<TA> v[kSlots];
#pragma unroll
            for (int j = 0; j < kSlots; ++j)
                if (pos[j] >= 0) v[j].load(y + (int64_t)pos[j] * H + c);
#pragma unroll
            for (int j = 0; j < kSlots; ++j) {
                if (pos[j] < 0) continue;  // contributes nothing
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
}

template <typename TA>
static cudaError_t launch_combine_t(const void* y_pairs, const float* topk_w, const int32_t* pair_pos, const void* y_shared,
                                    void* out, int T, int k, int H, cudaStream_t stream) {
    const int parts = (H / 8 + kCombineThreads - 1) / kCombineThreads;
    const int fill = (kBlocksPerSm * sm_count() + T - 1) / T;  // blocks per token that fill the SMs
    const dim3 grid((unsigned)T, (unsigned)(fill < parts ? fill : parts));
    constexpr int kMost = sizeof(TA) == 2 ? 8 : 4;
    auto kernel = k <= 1 ? combine_kernel<TA, 1> : k <= 2 ? combine_kernel<TA, 2> : k <= 4 ? combine_kernel<TA, 4> : combine_kernel<TA, kMost>;
    return launch_k(kernel, grid, dim3(kCombineThreads), 0, stream, static_cast<const TA*>(y_pairs), topk_w, pair_pos,
                    static_cast<const TA*>(y_shared), static_cast<TA*>(out), k, H);
}

cudaError_t launch_combine(const void* y_pairs, const float* topk_w, const int32_t* pair_pos, const void* y_shared,
                           void* out, int T, int k, int H, int act_dtype, cudaStream_t stream) {
    if (T == 0) return cudaSuccess;
    auto launch = act_dtype == GBMOE_BF16 ? launch_combine_t<__nv_bfloat16> : launch_combine_t<float>;
    return launch(y_pairs, topk_w, pair_pos, y_shared, out, T, k, H, stream);
}

}  // namespace gbmoe
