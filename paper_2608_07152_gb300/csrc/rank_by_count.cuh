// The order of a few thousand distinct 64-bit keys by counting: a key's
// position in the descending order is the number of larger keys.  Every
// block takes 32 keys, one a lane, and its warps a share of all keys each,
// staged in shared memory and read by every lane at once.  n^2 comparisons on
// every SM, and no chain of steps: 1,000 keys take 5 us and 8,192 25 us, where one
// block's sorting network took 11 and 65 us.
#pragma once

#include <cstdint>

namespace pvs {

constexpr int kRankWarps = 8;
constexpr int kRankKeys = 32;      // keys a block places
constexpr int kRankStage = 2048;   // keys staged at a time (16 KB)

struct RankShared {
    alignas(16) uint64_t keys[kRankStage];
    int larger[kRankKeys];
};

// The position of keys[blockIdx.x * kRankKeys + lane] among the n keys, the
// same in every warp of the block (kRankWarps * 32 threads; all of them call).
// `key` returns that key (0, which no key is, past the end).
__device__ __forceinline__ int position_by_count(const uint64_t* __restrict__ keys, int n,
                                                 RankShared& sh, uint64_t& key) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * kRankKeys + lane;
    key = i < n ? keys[i] : 0ull;
    if (threadIdx.x < kRankKeys) sh.larger[threadIdx.x] = 0;
    int count = 0;
    for (int base = 0; base < n; base += kRankStage) {
        const int m = min(kRankStage, n - base);
        for (int j = threadIdx.x; j < ((m + 1) & ~1); j += blockDim.x)
            sh.keys[j] = j < m ? keys[base + j] : 0ull;   // 0: larger than no key
        __syncthreads();
        const ulonglong2* s2 = reinterpret_cast<const ulonglong2*>(sh.keys);
#pragma unroll 4
        for (int j = warp; 2 * j < m; j += kRankWarps) {
            const ulonglong2 x = s2[j];
            count += (x.x > key) + (x.y > key);
        }
        __syncthreads();
    }
    atomicAdd(&sh.larger[lane], count);
    __syncthreads();
    return sh.larger[lane];
}

}  // namespace pvs
