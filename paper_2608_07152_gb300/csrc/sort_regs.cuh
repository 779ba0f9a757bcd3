// Descending sort of 64-bit keys by one CTA of 1,024 threads, in registers.
#pragma once

#include <cstdint>

namespace pvs {

constexpr int kSortThreads = 1024;

// At most 1024 E keys, E per thread: a bitonic network over the positions
// t E + e, whose strides under E stay within a thread, those under 32 E are
// shuffles within a warp, and only the rest go through shared memory (sk:
// 1024 E keys).  On entry the keys may sit anywhere; on return thread t holds
// the positions t E .. t E + E - 1 of the sorted order.
template <int E>
__device__ __forceinline__ void sort_desc(uint64_t (&v)[E], uint64_t* sk) {
    const int t = threadIdx.x;
    auto keep = [](uint64_t& a, uint64_t b, int i, int s, int size) {
        const bool keep_max = ((i & s) == 0) == ((i & size) == 0);
        a = keep_max ? (a > b ? a : b) : (a < b ? a : b);
    };
#pragma unroll 1
    for (int size = 2; size <= 1024 * E; size <<= 1) {
#pragma unroll 1
        for (int s = size >> 1; s >= 32 * E; s >>= 1) {   // another warp's element
            // element e of thread t at e 1024 + t: no bank conflicts
#pragma unroll
            for (int e = 0; e < E; ++e) sk[e * kSortThreads + t] = v[e];
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e)
                keep(v[e], sk[e * kSortThreads + (t ^ (s / E))], t * E + e, s, size);
            __syncthreads();
        }
#pragma unroll 1
        for (int s = min(size >> 1, 16 * E); s >= E; s >>= 1) {   // another lane's
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint64_t w = __shfl_xor_sync(0xffffffffu, v[e], s / E);
                keep(v[e], w, t * E + e, s, size);
            }
        }
#pragma unroll
        for (int s = E / 2; s > 0; s >>= 1) {   // this thread's
            if (s >= size) continue;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e & s) continue;
                const bool desc = ((t * E + e) & size) == 0;
                const uint64_t a = v[e], b = v[e | s];
                const bool swap = (a < b) == desc;
                v[e] = swap ? b : a;
                v[e | s] = swap ? a : b;
            }
        }
    }
}

}  // namespace pvs
