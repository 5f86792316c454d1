// Fused MoE, grouping step: stable counting sort of the (token, slot) pairs
// by expert. Three small kernels: per-block histograms, one scan that turns
// them into counts, offsets and per-block bases, and a scatter that ranks
// pairs inside a block in pair order (warp match + a prefix over the warps'
// counts), so the result is the stable order whatever the scheduling.
// Up to 1024 pairs (decode) all three steps run in one CTA. A pair whose
// expert id is outside [0, E) is dropped: pair_pos[p] = -1, and the sorted
// positions past the last kept pair hold -1.
#include "common.cuh"
#include "kernels.h"

namespace gbmoe {

constexpr int kPermBlock = 1024;  // pairs per block (one per thread)

int permute_blocks(int64_t P) { return (int)((P + kPermBlock - 1) / kPermBlock); }

// block histograms [nblk][E] + per-block bases [nblk][E]
size_t permute_scratch_ints(int64_t P, int E) { return 2 * (size_t)permute_blocks(P) * E; }

__global__ void __launch_bounds__(kPermBlock)
perm_hist_kernel(const int32_t* __restrict__ ids, int64_t P, int E, int32_t* __restrict__ block_hist) {
    pdl_enter();
    extern __shared__ int32_t s_hist[];
    for (int e = threadIdx.x; e < E; e += blockDim.x) s_hist[e] = 0;
    __syncthreads();
    int64_t p = (int64_t)blockIdx.x * kPermBlock + threadIdx.x;
    if (p < P) {
        const int e = ids[p];
        if (e >= 0 && e < E) atomicAdd(&s_hist[e], 1);  // out-of-range ids are dropped
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x) block_hist[(size_t)blockIdx.x * E + e] = s_hist[e];
}

// One block, thread e owns expert e: walks the block histograms in order.
// block_base receives the pairs of e in earlier blocks (the scatter adds e's
// offset).
__global__ void __launch_bounds__(512)
perm_scan_kernel(const int32_t* __restrict__ block_hist, int nblk, int E, int32_t* __restrict__ counts,
                 int32_t* __restrict__ offsets, int32_t* __restrict__ block_base) {
    pdl_enter();
    __shared__ int32_t s_warp[16];
    const int e = threadIdx.x;
    int run = 0;
    if (e < E)
        for (int b0 = 0; b0 < nblk; b0 += 8) {  // eight blocks' loads in flight
            int h[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) h[u] = b0 + u < nblk ? block_hist[(size_t)(b0 + u) * E + e] : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (b0 + u < nblk) block_base[(size_t)(b0 + u) * E + e] = run;
                run += h[u];
            }
        }
    // exclusive scan of the counts over experts
    const int lane = e & 31, warp = e >> 5;
    int v = (e < E) ? run : 0, incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0, wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            int o = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += o;
        }
        if (lane < 16) s_warp[lane] = wi - w;  // exclusive warp prefix
    }
    __syncthreads();
    int excl = s_warp[warp] + incl - v;
    if (e < E) {
        counts[e] = run;
        offsets[e] = excl;
        if (e == E - 1) offsets[E] = excl + run;
    }
}

// Place of this thread's pair among the block's pairs of the same expert, in
// pair order: the pairs of earlier warps, counted in s_cnt [warps][E] (which
// must be zero), plus those of earlier lanes. Three barriers, where warps
// taking turns needed one per warp (8192 x 8 pairs: 15.5 -> 5.0 us). Afterwards
// s_cnt[warps - 1][e] + the last warp's own count is the block's total of e.
__device__ __forceinline__ int block_rank(int e, bool valid, int E, uint16_t* s_cnt, int warps) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = valid ? e : -1 - lane;  // invalid lanes never match a real expert
    const uint32_t peers = __match_any_sync(0xffffffffu, m);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) s_cnt[warp * E + e] = (uint16_t)__popc(peers);
    __syncthreads();
    for (int x = threadIdx.x; x < E; x += blockDim.x) {  // exclusive prefix over the warps
        int run = 0;
#pragma unroll 8
        for (int w = 0; w < warps; ++w) {
            const int c = s_cnt[w * E + x];
            s_cnt[w * E + x] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
    return valid ? s_cnt[warp * E + e] + rank : 0;
}

__global__ void __launch_bounds__(kPermBlock)
perm_scatter_kernel(const int32_t* __restrict__ ids, int64_t P, int E, const int32_t* __restrict__ block_base,
                    const int32_t* __restrict__ offsets, int32_t* __restrict__ sorted_pair,
                    int32_t* __restrict__ pair_pos) {
    pdl_enter();
    extern __shared__ uint16_t s_cnt[];  // [kPermBlock / 32][E]
    const int warps = kPermBlock / 32;
    for (int i = threadIdx.x; i < warps * E; i += blockDim.x) s_cnt[i] = 0;
    const int64_t p = (int64_t)blockIdx.x * kPermBlock + threadIdx.x;
    const int id = p < P ? ids[p] : -1;
    const bool valid = id >= 0 && id < E;
    int base = 0;
    if (valid) base = offsets[id] + block_base[(size_t)blockIdx.x * E + id];
    const int kept = offsets[E];
    __syncthreads();
    const int pos = base + block_rank(id, valid, E, s_cnt, warps);
    if (valid) {
        sorted_pair[pos] = (int32_t)p;
        pair_pos[p] = pos;
    } else if (p < P) {
        pair_pos[p] = -1;  // dropped pair: no slot
    }
    // positions past the last kept pair (only when pairs were dropped) hold -1
    if (p < P && p >= kept) sorted_pair[p] = -1;
}

// P <= kPermBlock: histogram, scan and stable scatter in one CTA (one pair
// per thread). Same order and outputs as the three kernels above with one
// block: the block base of expert e is its offset.
__global__ void __launch_bounds__(kPermBlock)
perm_small_kernel(const int32_t* __restrict__ ids, int64_t P, int E, int32_t* __restrict__ counts,
                  int32_t* __restrict__ offsets, int32_t* __restrict__ sorted_pair, int32_t* __restrict__ pair_pos) {
    pdl_enter();
    extern __shared__ uint16_t s_cnt[];  // [warps that hold pairs][E], then E ints: counts, then offsets
    __shared__ int32_t s_warp[kPermBlock / 32];
    __shared__ int32_t s_kept;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int warps = (int)((P + 31) / 32);
    int32_t* s_off = reinterpret_cast<int32_t*>(s_cnt + warps * E + (warps * E & 1));
    for (int i = threadIdx.x; i < warps * E; i += blockDim.x) s_cnt[i] = 0;
    for (int i = threadIdx.x; i < E; i += blockDim.x) s_off[i] = 0;
    const int p = threadIdx.x;
    const int id = p < P ? ids[p] : -1;
    const bool valid = id >= 0 && id < E;  // out-of-range ids are dropped
    __syncthreads();
    if (valid) atomicAdd(&s_off[id], 1);
    const int rank = block_rank(id, valid, E, s_cnt, warps);  // (its barriers order the counts too)
    // exclusive scan of the counts over experts (thread e owns expert e; E <= 512)
    const int cnt = threadIdx.x < E ? s_off[threadIdx.x] : 0;
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = s_warp[lane], wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            int o = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += o;
        }
        s_warp[lane] = wi - w;  // exclusive warp prefix
    }
    __syncthreads();
    const int excl = s_warp[warp] + incl - cnt;
    if (threadIdx.x < E) {
        counts[threadIdx.x] = cnt;
        offsets[threadIdx.x] = excl;
        if (threadIdx.x == E - 1) {
            offsets[E] = excl + cnt;
            s_kept = excl + cnt;
        }
        s_off[threadIdx.x] = excl;
    }
    __syncthreads();
    if (valid) {
        const int pos = s_off[id] + rank;
        sorted_pair[pos] = p;
        pair_pos[p] = pos;
    } else if (p < P) {
        pair_pos[p] = -1;  // dropped pair: no slot
    }
    if (p < P && p >= s_kept) sorted_pair[p] = -1;  // past the last kept pair
}

// shared memory of the kernels above: at most 34 KB (E <= 512), within the
// default limit
static size_t small_smem(int64_t P, int E) {
    const size_t n = (size_t)((P + 31) / 32) * E;
    return (n + (n & 1)) * sizeof(uint16_t) + (size_t)E * sizeof(int32_t);
}

cudaError_t launch_permute(const int32_t* topk_ids, int64_t P, int E, int32_t* counts, int32_t* offsets,
                           int32_t* sorted_pair, int32_t* pair_pos, int32_t* scratch, cudaStream_t stream) {
    const int nblk = permute_blocks(P);
    if (nblk == 1)
        return launch_k(perm_small_kernel, dim3(1), dim3(kPermBlock), small_smem(P, E), stream, topk_ids, P, E,
                        counts, offsets, sorted_pair, pair_pos);
    int32_t* block_hist = scratch;
    int32_t* block_base = scratch + (size_t)nblk * E;
    if (nblk > 0) {
        if (const cudaError_t le = launch_k(perm_hist_kernel, dim3(nblk), dim3(kPermBlock), E * sizeof(int32_t),
                stream, topk_ids, P, E, block_hist); le != cudaSuccess)
            return le;
        cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    if (const cudaError_t le = launch_k(perm_scan_kernel, dim3(1), dim3(512), 0, stream, block_hist, nblk, E,
            counts, offsets, block_base); le != cudaSuccess)
        return le;
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || nblk == 0) return err;
    if (const cudaError_t le = launch_k(perm_scatter_kernel, dim3(nblk), dim3(kPermBlock),
            (size_t)(kPermBlock / 32) * E * sizeof(uint16_t), stream, topk_ids, P, E, block_base, offsets, sorted_pair, pair_pos); le != cudaSuccess)
        return le;
    return cudaGetLastError();
}

}  // namespace gbmoe
