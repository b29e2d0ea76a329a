// What the kernels that make sort keys share with the radix sort (scan.cu):
// the digit histogram of the keys and the clearing of the sort's tile records,
// done while the keys are made, so that the sort is its passes alone.
#pragma once

#include "common.cuh"

namespace rk {

constexpr int RAD_T = 256;
constexpr int RAD_PASSES = 4;                    // 8-bit digits of a 32-bit key
constexpr int RAD_TILE_MIN = 2048;               // smallest tile of a pass (records are sized for it)

// The sort's scratch: per-pass digit counts, tile counters, and the tiles'
// look-back records.
struct RadixWs {
    unsigned long long* counts;    // [RAD_PASSES][256]
    int* ctr;                      // [RAD_PASSES] tiles handed out
    unsigned long long* status;    // [passes][tiles][256]
    long long n_status;            // words of status that this sort uses
    int npass;
};

// Adds the digits of one key per lane (FULL warps) to the block's histogram.  A
// warp whose keys share a digit, the rule for the upper ones, adds it once.
__device__ __forceinline__ void radix_count(uint32_t key, bool valid, int npass, int (*hist)[256]) {
    const unsigned live = __ballot_sync(0xffffffffu, valid);
    if (!live) return;
    const uint32_t k0 = __shfl_sync(0xffffffffu, key, __ffs(live) - 1);
    const uint32_t diff = __reduce_or_sync(0xffffffffu, valid ? key ^ k0 : 0u);
    const bool first = (threadIdx.x & 31) == (unsigned)(__ffs(live) - 1);
    for (int p = 0; p < npass; ++p) {
        if (((diff >> (8 * p)) & 255u) == 0u) {
            if (first) atomicAdd(&hist[p][(k0 >> (8 * p)) & 255u], __popc(live));
        } else if (valid) {
            atomicAdd(&hist[p][(key >> (8 * p)) & 255u], 1);
        }
    }
}

// Block end: the histogram into the global counts (blockDim.x == RAD_T, after
// a __syncthreads), and this block's share of the tile records cleared.
__device__ __forceinline__ void radix_finish(const RadixWs& ws, int (*hist)[256]) {
    for (int p = 0; p < ws.npass; ++p) {
        const int c = hist[p][threadIdx.x];
        if (c) atomicAdd(&ws.counts[256 * p + threadIdx.x], (unsigned long long)c);
    }
    for (long long i = blockIdx.x * (long long)RAD_T + threadIdx.x; i < ws.n_status; i += (long long)gridDim.x * RAD_T)
        ws.status[i] = 0ull;
}

// Rounds of 256 keys a block of a key kernel takes: up to 8, as long as a few
// blocks are left for every SM.
inline int radix_rounds(long long n, int num_sms) {
    const long long r = n / (256LL * 4 * num_sms);
    return r < 1 ? 1 : (r > 8 ? 8 : (int)r);
}

}  // namespace rk
