// pvs_rank_exact_noalloc: exact top-n ranking of a caller-held set of vectors
// that performs no device memory allocation.
//
// It is the score-key-sort part of a pull (exact scores -> 64-bit rank keys
// -> descending sort -> emit), run over vectors the caller already holds on
// the device, with the rank keys kept in one file-scope static device array
// instead of memory obtained from cudaMalloc.  Some callers cannot allocate
// device memory at the point where they need a ranking: services whose
// device memory is owned by their own pool or budget, where an allocation
// outside the pool either fails or breaks its accounting, and
// latency-critical callers, for whom cudaMalloc can take milliseconds and
// cudaFree waits for the whole device to go idle.
//
// The scratch array: PVS_NOALLOC_MAX_VECTORS 64-bit keys plus one status word
// (64 KiB + 256 B).  Every GPU that loads this library holds it until the
// process exits.  Every call on a device uses the same array and leaves its
// keys behind; the status word is cleared at the start of each call, and no
// key is read that the same call did not write.  Calls whose device work
// overlaps (for example on two streams at once) race on the array.
//
// Host code must not use the array's name as a device address: the symbol is
// a host-side stand-in.  The device address is fetched once per device with
// cudaGetSymbolAddress, during the first call made with that device current.
// That first call should therefore come before any stream capture begins.
#include <mutex>

#include "exact_dot.cuh"
#include "kernels.h"
#include "pvs_common.cuh"
#include "rank_by_count.cuh"

namespace pvs {

constexpr int kNoAllocMax = PVS_NOALLOC_MAX_VECTORS;
constexpr int kNoAllocStatusSlot = kNoAllocMax;            // key slots, then the status
constexpr int kNoAllocSlots = kNoAllocMax + 32;           // 256 B of status padding

static __device__ __align__(256) unsigned long long g_noalloc_scratch[kNoAllocSlots];

// The rare rows the float32 decision leaves open, out of line.
static __device__ __noinline__ float exact_dot_open(const float* __restrict__ q,
                                                    const float* __restrict__ v, int dim) {
    bool fb;
    return exact_dot_warp_any(q, v, dim, &fb);
}

// One warp per vector: finite check, exact score, rank key into scratch; four
// warps a block, so that a thousand vectors reach every SM.
// VEC: 16-byte loads (query and vectors aligned, dim a multiple of 4), else
// scalar ones.  Bound by latency: one round trip to memory, a chain of products
// per accumulator, five merges.  In binary64 (1/64 of the float32 rate), with
// a pass of its own for the finite check, 1,000 x 768 took 37 us; now 4.6 us.
constexpr int kScoreWarps = 4;
template <bool VEC>
__global__ void __launch_bounds__(kScoreWarps * 32) noalloc_score_kernel(
    const float* __restrict__ q, const float* __restrict__ vecs, int n, int dim,
    unsigned long long* scratch) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kScoreWarps + (threadIdx.x >> 5);
    if (i >= n) return;
    const float* v = vecs + (int64_t)i * dim;
    EftAcc acc, acc2;   // two dependency chains, merged as in the butterfly
    bool finite = true;
    if constexpr (VEC) {
        const float4* q4 = reinterpret_cast<const float4*>(q);
        const float4* v4 = reinterpret_cast<const float4*>(v);
        constexpr int kBatch = 6;
        const int n4 = dim >> 2;
        for (int j0 = lane; j0 < n4; j0 += kWarp * kBatch) {
            float4 x[kBatch], y[kBatch];
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int j = j0 + kWarp * b;
                x[b] = y[b] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (j < n4) {
                    y[b] = __ldg(v4 + j);
                    x[b] = __ldg(q4 + j);
                }
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                finite &= isfinite(x[b].x) && isfinite(x[b].y) && isfinite(x[b].z) &&
                          isfinite(x[b].w) && isfinite(y[b].x) && isfinite(y[b].y) &&
                          isfinite(y[b].z) && isfinite(y[b].w);
                acc.add_product(x[b].x, y[b].x);
                acc2.add_product(x[b].y, y[b].y);
                acc.add_product(x[b].z, y[b].z);
                acc2.add_product(x[b].w, y[b].w);
            }
        }
    } else {
        constexpr int kBatch = 8;
        for (int j0 = lane; j0 < dim; j0 += kWarp * kBatch) {
            float x[kBatch], y[kBatch];
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int j = j0 + kWarp * b;
                y[b] = j < dim ? __ldg(v + j) : 0.0f;
                x[b] = j < dim ? __ldg(q + j) : 0.0f;
            }
#pragma unroll
            for (int b = 0; b < kBatch; b += 2) {
                finite &= isfinite(x[b]) && isfinite(y[b]) && isfinite(x[b + 1]) &&
                          isfinite(y[b + 1]);
                acc.add_product(x[b], y[b]);
                acc2.add_product(x[b + 1], y[b + 1]);
            }
        }
    }
    finite = __all_sync(0xffffffffu, finite);
    int* status = reinterpret_cast<int*>(scratch + kNoAllocStatusSlot);
    if (!finite) {
        if (lane == 0) {
            set_status(status, PVS_ERR_NONFINITE);
            scratch[i] = 0ull;
        }
        return;
    }
    acc.merge(acc2.s, acc2.c, acc2.a1, acc2.a2);
    float s;
    if (!eft_finish(acc, dim, &s)) s = exact_dot_open(q, v, dim);
    if (lane == 0) {
        if (!isfinite(s)) set_status(status, PVS_ERR_OVERFLOW);
        scratch[i] = rank_key(s, (uint32_t)i);
    }
}

__global__ void __launch_bounds__(kRankWarps * 32) noalloc_rank_emit_kernel(
    const unsigned long long* __restrict__ scratch, int n, int top, int64_t* out_ids,
    float* out_scores) {
    __shared__ RankShared sh;
    uint64_t key;
    const int r = position_by_count(reinterpret_cast<const uint64_t*>(scratch), n, sh, key);
    if (threadIdx.x < kRankKeys && blockIdx.x * kRankKeys + threadIdx.x < n && r < top) {
        out_ids[r] = rank_key_id(key);
        out_scores[r] = rank_key_score(key);
    }
}

namespace {

constexpr int kMaxDevices = 256;
std::mutex g_setup_mutex;
unsigned long long* g_scratch_addr[kMaxDevices] = {nullptr};

// Device address of the scratch array for the current device (set up once).
cudaError_t scratch_address(unsigned long long** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = static_cast<unsigned long long*>(p);
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

bool on_device(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace pvs

extern "C" pvs_status pvs_rank_exact_noalloc(const float* query, const float* vecs, int32_t n,
                                             int32_t dim, int32_t top, int64_t* out_ids,
                                             float* out_scores, void* cuda_stream) {
    using namespace pvs;
    if (n < 0 || n > kNoAllocMax || dim < 1 || dim > kMaxDim || top < 0 || top > n)
        return PVS_ERR_INVALID;
    if (!query || !on_device(query)) return PVS_ERR_INVALID;
    if (n > 0 && (!vecs || !on_device(vecs))) return PVS_ERR_INVALID;
    if (top > 0 && (!out_ids || !out_scores || !on_device(out_ids) || !on_device(out_scores)))
        return PVS_ERR_INVALID;
    unsigned long long* scratch = nullptr;
    cudaError_t e = scratch_address(&scratch);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return PVS_ERR_CUDA;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    e = cudaMemsetAsync(scratch + kNoAllocStatusSlot, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess && n > 0) {
        count_launches(1);
        const bool vec = dim % 4 == 0 && ((reinterpret_cast<uintptr_t>(query) |
                                           reinterpret_cast<uintptr_t>(vecs)) & 15u) == 0;
        const int blocks = (n + kScoreWarps - 1) / kScoreWarps;
        if (vec)
            noalloc_score_kernel<true><<<blocks, kScoreWarps * 32, 0, st>>>(query, vecs, n, dim,
                                                                            scratch);
        else
            noalloc_score_kernel<false><<<blocks, kScoreWarps * 32, 0, st>>>(query, vecs, n, dim,
                                                                             scratch);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && top > 0) {
        count_launches(1);
        noalloc_rank_emit_kernel<<<(n + kRankKeys - 1) / kRankKeys, kRankWarps * 32, 0, st>>>(scratch, n, top,
                                                                            out_ids, out_scores);
        e = cudaGetLastError();
    }
    unsigned long long status = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&status, scratch + kNoAllocStatusSlot, sizeof(status),
                            cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return PVS_ERR_CUDA;
    }
    return (pvs_status)(int)(status & 0xffffffffull);
}
