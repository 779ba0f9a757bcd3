// The first pull of a lone cursor in four launches (Sec. 2.3.1 incremental
// ranking, Sec. 2.1 exact prefix): the first working set is the rows that can
// hold the next H ranks; all of them are scored exactly, and the first ranks
// come out in order.
//
//   1. first_threshold_kernel  a value v that at least H rows' lower bounds reach;
//   2. first_set_kernel        W = the live rows with hi >= v (unordered);
//   3. refine_ring_kernel      the exact score of every row of W, on every SM;
//   4. first_emit_kernel       W's certified rows ordered by rank key (score desc, id
//                              asc), the first n ranks written and marked (those
//                              above the first row that missed its interval).
// Every row outside W has hi < v, so the rows of W that score v or more, H at
// least, are the first ranks: all of them are certified, usually many more
// than H (intervals are wider than the spread of the best scores).  More than
// kFirstMax rows in W: steps 3 and 4 do nothing and the host goes through the
// ordered working set instead (build_working_set), whose later pulls score
// only what they need.
//
// Bound by latency: W is a few thousand rows.  The incremental path scored
// nearly all of W in its first pull anyway and needed ten launches for the
// working set and the first page, then a pull for every further 80 ranks.
#include "kernels.h"
#include "pvs_common.cuh"

namespace pvs {
namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 2048;
constexpr int kStageMax = 50 * 1024;   // values staged in shared memory (200 KB)

struct ThresholdShared {
    unsigned int hist[kBins];
    float red[kWarps][2];
    unsigned int warp_tot[kWarps];
    int bin;
    unsigned int above;   // entries in the bins past `bin`
    unsigned int inside;  // entries in it
};

// Block-wide (kThreads threads, after a barrier): a value v with at least k of
// the entries >= v, or -inf if there are fewer than k (-inf entries do not
// count): the smallest entry in the bins, linear in value, that hold the k
// largest.  The bin with the k-th largest is split again while it holds many
// entries, so few more than k reach v.  [vmin, vmax]: this thread's share of the
// entries' range.
__device__ __forceinline__ float block_floor(const float* src, int len, unsigned int k, float vmin,
                                             float vmax, ThresholdShared& sh) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    auto block_range = [&](float& mn, float& mx) {
        mx = warp_max(mx);
        mn = -warp_max(-mn);
        if (lane == 0) {
            sh.red[warp][0] = mn;
            sh.red[warp][1] = mx;
        }
        __syncthreads();
        mn = sh.red[lane][0];
        mx = sh.red[lane][1];
        mx = warp_max(mx);
        mn = -warp_max(-mn);
        __syncthreads();
    };
    block_range(vmin, vmax);
    if (!(vmin <= vmax)) return -INFINITY;   // no entry
    float floor_v = vmin;
    unsigned int above = 0;        // entries > the current range
    for (int round = 0; round < 3; ++round) {
        for (int i = t; i < kBins; i += kThreads) sh.hist[i] = 0;
        __syncthreads();
        const float base = vmin, scale = vmax > vmin ? (kBins - 0.5f) / (vmax - vmin) : 0.0f;
        const float top = vmax;
        auto bin_of = [&](float v) {   // monotone in v
            return min(kBins - 1, (int)((v - base) * scale));
        };
        uint32_t run_b = kBins, run_n = 0;   // runs of one bin counted in a register
        for (int i = t; i < len; i += kThreads) {
            const float v = src[i];
            if (!(v >= base && v <= top)) continue;
            const uint32_t b = (uint32_t)bin_of(v);
            if (b != run_b) {
                if (run_n) atomicAdd(&sh.hist[run_b], run_n);
                run_b = b;
                run_n = 0;
            }
            ++run_n;
        }
        if (run_n) atomicAdd(&sh.hist[run_b], run_n);
        __syncthreads();
        // the bin of the k-th largest: thread t holds bins 2 t and 2 t + 1
        const unsigned int h0 = sh.hist[2 * t], h1 = sh.hist[2 * t + 1];
        unsigned int incl = h0 + h1;   // suffix sums over the lanes, then the warps
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int v = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += v;
        }
        if (lane == 0) sh.warp_tot[warp] = incl;
        if (t == 0) sh.bin = -1;
        __syncthreads();
        unsigned int past = above;
        for (int w = warp + 1; w < kWarps; ++w) past += sh.warp_tot[w];
        const unsigned int past1 = past + incl - h0 - h1;   // entries past bin 2 t + 1
        const unsigned int past0 = past1 + h1;              // past bin 2 t
        if (past1 < k && k <= past1 + h1) {
            sh.bin = 2 * t + 1;
            sh.above = past1;
            sh.inside = h1;
        } else if (past0 < k && k <= past0 + h0) {
            sh.bin = 2 * t;
            sh.above = past0;
            sh.inside = h0;
        }
        __syncthreads();
        if (sh.bin < 0) return -INFINITY;   // fewer than k
        const int bin = sh.bin;
        const unsigned int inside = sh.inside;
        above = sh.above;
        // the range of the bin's entries
        float mn = INFINITY, mx = -INFINITY;
        for (int i = t; i < len; i += kThreads) {
            const float v = src[i];
            if (!(v >= base && v <= top) || bin_of(v) != bin) continue;
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
        block_range(mn, mx);
        floor_v = mn;
        vmin = mn;
        vmax = mx;
        if (inside <= 64 || inside <= k / 16 || !(vmin < vmax)) break;
    }
    return floor_v;
}

// One CTA.  A value that at least k live entries reach (sel->prefix = its key;
// 0, which every live row reaches, for k = 0 or fewer than k).  Also zeroes
// the cursor's working-set length and its frontier.
__global__ void __launch_bounds__(kThreads, 1)
    first_threshold_kernel(const float* __restrict__ vals, int len, unsigned int k,
                           SelectState* sel, DevCounters* ctr, int staged) {
    extern __shared__ float4 stage4[];
    __shared__ ThresholdShared sh;
    const int t = threadIdx.x;
    if (t == 0) {
        sel->prefix = 0;
        ctr->w_len = 0;
        ctr->cand = 0;   // the emission's blocks that are done
        ctr->front_k = 0;
        ctr->front_hint = 0;
    }
    if (k == 0) return;   // every live row
    float* st = reinterpret_cast<float*>(stage4);
    float vmin = INFINITY, vmax = -INFINITY;
    auto see = [&](float v) {
        if (v == -INFINITY) return;
        vmin = fminf(vmin, v);
        vmax = fmaxf(vmax, v);
    };
    if (staged) {
        const int n4 = len >> 2;
        const float4* v4 = reinterpret_cast<const float4*>(vals);
#pragma unroll 4
        for (int i = t; i < n4; i += kThreads) {
            const float4 v = v4[i];
            stage4[i] = v;
            see(v.x), see(v.y), see(v.z), see(v.w);
        }
        for (int i = 4 * n4 + t; i < len; i += kThreads) {
            st[i] = vals[i];
            see(st[i]);
        }
    } else {
        for (int i = t; i < len; i += kThreads) see(vals[i]);
    }
    __syncthreads();
    const float v = block_floor(staged ? st : vals, len, k, vmin, vmax, sh);
    if (t == 0 && v != -INFINITY) sel->prefix = fkey(v);
}

// W, unordered: the live rows that reach the threshold.  lo is -inf exactly
// where hi is; a threshold that is a finite bound's key needs hi alone, and 0
// (every live row) reads lo.
__global__ void __launch_bounds__(256) first_set_kernel(const float* __restrict__ lo,
                                                       const float* __restrict__ hi, int64_t rows,
                                                       const SelectState* sel, int32_t* w_id,
                                                       float* w_lo, float* w_hi,
                                                       unsigned int* w_len) {
    const uint32_t tau = (uint32_t)sel->prefix;
    const int lane = threadIdx.x & 31;
    const int64_t quads = (rows + 3) / 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float* src = tau ? hi : lo;
    // whole warps run every step
    for (int64_t g0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); g0 < quads;
         g0 += stride) {
        const int64_t r0 = 4 * (g0 + lane);
        float v[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (r0 + 3 < rows) {
            const float4 x = *reinterpret_cast<const float4*>(src + r0);
            v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
        } else {
            for (int j = 0; j < 4; ++j)
                if (r0 + j < rows) v[j] = src[r0 + j];
        }
        unsigned int take = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            take |= (unsigned int)(v[j] != -INFINITY && fkey(v[j]) >= tau) << j;
        if (!__any_sync(0xffffffffu, take != 0)) continue;
        const int mine = __popc(take);
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        unsigned int base = 0;
        if (lane == 31) base = atomicAdd(w_len, (unsigned int)incl);
        unsigned int at = __shfl_sync(0xffffffffu, base, 31) + (unsigned int)(incl - mine);
        for (int j = 0; j < 4; ++j) {
            if (!((take >> j) & 1u)) continue;
            w_id[at] = (int32_t)(r0 + j);
            w_lo[at] = lo[r0 + j];
            w_hi[at] = hi[r0 + j];
            ++at;
        }
    }
}

struct FirstEmitArgs {
    const int32_t* w_id;
    const float* w_lo;
    float* lo;
    float* hi;
    int n;                   // ranks to emit at most
    const SelectState* sel;  // the threshold: rows of its key and above are certified
    int64_t* out_ids;
    float* out_scores;
    DevCounters* ctr;
    const int* status;
    unsigned int* len_mirror;   // pinned: the working set's length, and the ranks emitted
    int* status_mirror;         // pinned: written last
};

__device__ __forceinline__ void emit_rank(const FirstEmitArgs& a, int r, uint64_t key) {
    const uint32_t id = rank_key_id(key);
    a.out_ids[r] = (int64_t)id;
    a.out_scores[r] = rank_key_score(key);
    a.lo[id] = -INFINITY;
    a.hi[id] = -INFINITY;
}

// Order the certified rows of the scored set and emit the first n.  A key's
// rank is the number of larger keys, and every key larger than a certified
// one is certified too: each block gathers the certified keys in shared memory
// and counts for its share of the set, 32 rows at a time, one a lane, its warps
// a part of the keys each.  The last block to finish publishes.  Bound by
// latency: one block that ranked by bins of the scores, or sorted where a
// bin was crowded, took 14 us at 2,200 rows and 24 to 45 us in clusters of near
// neighbours; now 11, and 12 to 15 us.
constexpr int kEmitWarps = 32;

__global__ void __launch_bounds__(kEmitWarps * 32, 1) first_emit_kernel(const FirstEmitArgs a) {
    extern __shared__ ulonglong2 emit_sh[];   // kFirstMax keys
    uint64_t* sk = reinterpret_cast<uint64_t*>(emit_sh);
    __shared__ unsigned int count;
    __shared__ unsigned int larger[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned int len = a.ctr->w_len;
    const bool fits = len <= (unsigned int)kFirstMax;
    const uint32_t tau = (uint32_t)a.sel->prefix;
    const uint64_t bad = a.ctr->bad_key;   // ranks from this key on are void (0: none)
    unsigned int m = 0;
    if (fits) {
        auto key_of = [&](unsigned int i) {
            return i < len ? rank_key(a.w_lo[i], (uint32_t)a.w_id[i]) : 0ull;
        };
        uint64_t next = key_of(blockIdx.x * 32u + lane);   // of this block's first rows
        if (t == 0) count = 0;
        __syncthreads();
        for (unsigned int i0 = warp * 32; i0 < len; i0 += kEmitWarps * 32) {
            const uint64_t key = key_of(i0 + lane);
            const bool take = key > bad && (uint32_t)(key >> 32) >= tau;
            const unsigned int bal = __ballot_sync(0xffffffffu, take);
            unsigned int base = 0;
            if (lane == 0 && bal) base = atomicAdd(&count, (unsigned int)__popc(bal));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (take) sk[base + __popc(bal & ((1u << lane) - 1u))] = key;
        }
        __syncthreads();
        m = count;
        if (t == 0 && (m & 1u)) sk[m] = 0ull;   // larger than no key (m < kFirstMax: it is odd)
        for (unsigned int i0 = blockIdx.x * 32u; i0 < len; i0 += gridDim.x * 32u) {
            const uint64_t key = next;
            next = key_of(i0 + gridDim.x * 32u + lane);
            const bool mine = key > bad && (uint32_t)(key >> 32) >= tau;
            if (t < 32) larger[t] = 0;
            __syncthreads();
            if (__any_sync(0xffffffffu, mine)) {   // the same in every warp
                unsigned int above = 0;
#pragma unroll 4
                for (unsigned int j = warp; 2 * j < m; j += kEmitWarps) {
                    const ulonglong2 x = emit_sh[j];
                    above += (x.x > key) + (x.y > key);
                }
                atomicAdd(&larger[lane], above);
            }
            __syncthreads();
            if (warp == 0 && mine && larger[lane] < (unsigned int)a.n)
                emit_rank(a, (int)larger[lane], key);
            __syncthreads();
        }
    }
    __threadfence_system();   // this thread's ranks, before the words below
    __syncthreads();
    if (t == 0 && atomicAdd(&a.ctr->cand, 1u) == gridDim.x - 1) {
        __threadfence_system();   // the other blocks' ranks
        a.ctr->cand = len;
        if (fits) a.ctr->cand_total += len;
        volatile unsigned int* words = a.len_mirror;
        words[0] = fits ? len : 0xffffffffu;   // (nothing emitted)
        words[1] = fits ? min(m, (unsigned int)a.n) : 0u;
        __threadfence_system();
        *reinterpret_cast<volatile int*>(a.status_mirror) =
            *reinterpret_cast<const volatile int*>(a.status);
    }
}

}  // namespace

bool first_threshold_fits(int64_t len) { return len > 0 && len <= kStageMax; }

cudaError_t launch_first_set(const FirstSetArgs& a, int num_sms, cudaStream_t st) {
    const bool staged = a.k > 0 && (reinterpret_cast<uintptr_t>(a.vals) & 15u) == 0;
    const size_t smem = staged ? (size_t)((a.len + 3) / 4) * sizeof(float4) : 0;
    if (smem > 0) {
        cudaError_t e = raise_smem_limit((const void*)first_threshold_kernel, smem);
        if (e != cudaSuccess) return e;
    }
    count_launches(2);
    first_threshold_kernel<<<1, kThreads, smem, st>>>(a.vals, (int)a.len, (unsigned int)a.k, a.sel,
                                                      a.ctr, staged ? 1 : 0);
    int64_t blocks = (a.rows / 4 + 255) / 256 + 1;
    if (blocks > 8 * (int64_t)num_sms) blocks = 8 * (int64_t)num_sms;
    first_set_kernel<<<(unsigned)blocks, 256, 0, st>>>(a.lo, a.hi, a.rows, a.sel, a.w_id, a.w_lo,
                                                       a.w_hi, &a.ctr->w_len);
    return cudaGetLastError();
}

cudaError_t launch_first_emit(const FirstSetArgs& a, int n, int64_t* out_ids, float* out_scores,
                              const int* status, unsigned int* len_mirror, int* status_mirror,
                              int num_sms, cudaStream_t st) {
    constexpr size_t smem = (size_t)kFirstMax * sizeof(uint64_t);
    cudaError_t e = raise_smem_limit((const void*)first_emit_kernel, smem);
    if (e != cudaSuccess) return e;
    const FirstEmitArgs f{a.w_id, a.w_lo, a.lo, a.hi, n, a.sel, out_ids, out_scores, a.ctr, status,
                          len_mirror, status_mirror};
    count_launches(1);
    first_emit_kernel<<<num_sms, kEmitWarps * 32, smem, st>>>(f);
    return cudaGetLastError();
}

}  // namespace pvs
