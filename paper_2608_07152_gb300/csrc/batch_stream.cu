// Batched PVS interval pass that streams the Int8 codes themselves through the
// tensor cores (Sec. 2.3.1 intervals for many queries at once; App. A.1 bound
// arithmetic): up to kStreamQueries queries per pass, one read of the codes.
//
// D[rows x Qp] = A[rows x m] * B[Qp x m]^T with A and B the exact Int8 codes as
// f16 (|z| <= 127, products below 2^14, partial sums below 2^24: fp32
// accumulation is exact).  GB300 has no Int8 tcgen05 MMA and f16 codes in HBM
// would double the bytes, so the codes stay Int8 until they are on the SM:
//
//   CTA pairs (cta_group::2, M = 256): each CTA owns 128 rows of the pair's
//   tile, and half of the queries (B), resident in its shared memory for the
//   whole pass.  18 warps per CTA:
//   warp 0      TMA producer: boxes of 128 rows x 128 code bytes into a ring
//               (128-byte swizzle, L2 evict-first);
//   warp 1      allocates TMEM; in the even CTA one thread issues the pair's
//               MMAs (M = 256, N = Qp, K = 16) with A read from TMEM and B from
//               shared memory;
//   warps 2-9   converters: a thread owns a row (= a TMEM lane), reads its 128
//               bytes of a box, widens them to f16 in registers (exact) and
//               stores them as the A operand in TMEM; two groups of four warps
//               take alternate boxes (full barriers of ring_turns.h: the ring
//               has seven buffers at 768 bytes and 128 queries).  A box is
//               handed over in two halves (32 columns each, eight buffers):
//               the loop converter -> issuer -> MMA -> commit -> converter
//               crosses the pair twice and takes thousands of cycles, so many
//               small buffers keep the MMAs fed;
//   warps 10-17 epilogue: one row per thread, 32 query columns per
//               tcgen05.ld, two queries per f32x2 instruction; two
//               accumulators let it run under the next tile's MMAs.
//
// Operand bytes per tile and SM: 128 m from HBM once, B never again.  The
// bf16 pass (batch_gemm.cu) reads 2 m per row from HBM and fetches B from L2
// for every tile; it serves row widths this kernel has no room for.
//
// Modes:
//   sample  lower bounds of every tile_stride-th tile: one float per row, or that of the
//           row of the largest centre among 32 (a distinct row's bound either way, so the
//           k-th largest stored never exceeds the k-th largest lower bound);
//   filter  rows whose upper bound reaches the query's threshold tau_q are
//           appended to its working set, rows whose lower bound does are
//           counted.  One FMA per pair and a three-input maximum reject nearly all
//           of them: dot * s_v < theta_q implies hi < tau_q
//           (stream_theta_kernel).  A survivor is a record (row, query, dot) in its
//           warp's buffer; 32 records at a time, one per lane, get their interval and
//           their place (reserving places chunk by chunk waited out an atomic's
//           round trip for each).
#include <mutex>

#include "f32x2.cuh"
#include "kernels.h"
#include "pvs_common.cuh"
#include "ring_turns.h"
#include "tc.cuh"
#include "tensor_map.h"

namespace pvs {
namespace {

constexpr int kRows = 128;                    // rows per tile and CTA
constexpr int kBox = 128;                     // code bytes per row and box
constexpr int kBoxBytes = kRows * kBox;       // 16 KB
constexpr int kMaxStages = 8;
constexpr int kABufs = 8;                     // TMEM buffers of half a widened box
constexpr int kABufCols = kBox / 4;           // two f16 per 32-bit column
constexpr int kRecords = 160;                 // survivors buffered per epilogue warp
constexpr int kAccCols = kStreamQueries;      // columns of one accumulator
constexpr uint32_t kTmemCols = 512;
static_assert(2 * kAccCols + kABufs * kABufCols <= (int)kTmemCols, "TMEM columns");
constexpr int kConvWarps = 8, kEpiWarps = 8;
constexpr int kStreamThreads = (2 + kConvWarps + kEpiWarps) * 32;
constexpr int kSmemMax = 226 * 1024;

struct StreamShared {
    uint64_t full[2 * kMaxStages];   // TMA -> converters (ring_turns.h)
    uint64_t empty[kMaxStages];   // converters -> TMA
    uint64_t afull[kABufs];       // both CTAs' converters -> MMA (even CTA)
    uint64_t aempty[kABufs];      // MMA -> converters (both CTAs)
    uint64_t tfull[2];            // MMA -> epilogue (both CTAs)
    uint64_t tempty[2];           // both CTAs' epilogues -> MMA (even CTA)
    uint64_t bfull;               // both CTAs' B bytes (even CTA)
    uint64_t drained;             // every MMA issued has completed (both CTAs)
    uint32_t tmem_base;
    int abort;
    QueryScalars qs[kStreamQueries];
    alignas(16) float ntheta[kStreamQueries];   // -theta_q
    alignas(16) float tau[kStreamQueries];
    uint2 rec[kEpiWarps][kRecords];             // (row, query << 25 | dot)
};

__device__ __forceinline__ bool aborted(StreamShared& sh) {
    return *reinterpret_cast<volatile int*>(&sh.abort) != 0;
}
// A wait gave up: recorded, and the other roles of this CTA stop at their next check.
__device__ __forceinline__ void give_up(StreamShared& sh, int* status) {
    set_status(status, PVS_ERR_TIMEOUT);
    *reinterpret_cast<volatile int*>(&sh.abort) = 1;
}

// The 16 codes of a 16-byte piece -> 8 registers, in order.
__device__ __forceinline__ void widen16(const uint4& v, uint32_t* f) {
    codes_to_f16x2(v.x, f[0], f[1]);
    codes_to_f16x2(v.y, f[2], f[3]);
    codes_to_f16x2(v.z, f[4], f[5]);
    codes_to_f16x2(v.w, f[6], f[7]);
}

__device__ __forceinline__ float max3_of(float m, uint64_t v) {
    float x, y;
    f2_unpack(v, x, y);
    return fmaxf(fmaxf(m, x), y);
}

// Every CTA of a pair runs the same number of tile slots; a slot past the last
// tile loads boxes out of range (zero fill) and writes nothing.
// kBounds: both bounds of every row (a.dump_hi), for diagnostics; apart, since the
// branch in the serving kernel cost its filter up to 5% (1M x 384 118 -> 124 us).
template <bool kBounds>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kStreamThreads, 1)
    batch_stream_kernel(const __grid_constant__ CUtensorMap tmA,
                        const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ StreamArgs a, int stages) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t* bsm = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
    const int bhalf = a.nq_pad / 2;                 // query rows of B in this CTA
    const int kchunks = a.m_pad / 64;               // B: [kchunks][bhalf][64 f16], swizzled
    uint8_t* ring = bsm + (size_t)kchunks * bhalf * 128;
    StreamShared& sh = *reinterpret_cast<StreamShared*>(ring + (size_t)stages * kBoxBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int boxes = (a.m_pad + kBox - 1) / kBox;  // per tile
    const int64_t ntiles = (a.rows + kRows - 1) / kRows;
    const int64_t niter = (ntiles + a.tile_stride - 1) / a.tile_stride;
    const uint32_t crank = cluster_ctarank();
    const bool leader = crank == 0;
    const int64_t slot0 = blockIdx.x / 2, nslots = gridDim.x / 2;
    const int bars = turn_bars(stages);             // full barriers of the ring
    // tile slots of this pair: slot0, slot0 + nslots, ... while 2 t < niter
    const int64_t pair_tiles = (niter + 1) / 2;
    const int nmine = slot0 < pair_tiles ? (int)((pair_tiles - slot0 + nslots - 1) / nslots) : 0;

    for (int i = threadIdx.x; i < kStreamQueries; i += blockDim.x) {
        const bool on = i < a.nq && a.qs[i].status == 0;
        sh.qs[i] = on ? a.qs[i] : QueryScalars{};
        // padding columns, and queries the encoder refused, are never candidates
        sh.ntheta[i] = on ? (a.theta ? -a.theta[i] : INFINITY) : -INFINITY;
        sh.tau[i] = on && a.tau ? a.tau[i] : INFINITY;
    }
    if (threadIdx.x == 0) {
        for (int f = 0; f < bars; ++f) mbar_init(&sh.full[f], 1);
        for (int s = 0; s < stages; ++s) mbar_init(&sh.empty[s], 4);   // one converter group
        for (int b = 0; b < kABufs; ++b) {
            mbar_init(&sh.afull[b], 8);                  // one group of each CTA
            mbar_init(&sh.aempty[b], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sh.tfull[b], 1);
            mbar_init(&sh.tempty[b], 2 * kEpiWarps);     // both CTAs' epilogues
        }
        mbar_init(&sh.bfull, 1);
        mbar_init(&sh.drained, 1);
        sh.abort = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tc::tmem_alloc_pair(&sh.tmem_base, kTmemCols);
        tc::fence_before_sync();
    }
    __syncthreads();
    cluster_barrier();   // both CTAs' barriers and TMEM are ready
    tc::fence_after_sync();
    const uint32_t tmem = sh.tmem_base;
    const uint32_t tmem_a = tmem + 2 * kAccCols;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0 && nmine > 0) {
            tc::prefetch_tmap(&tmA);
            tc::prefetch_tmap(&tmB);
            const uint64_t pol = l2_evict_first_policy();
            // B once: the bytes of both CTAs are counted on the even CTA's barrier
            if (leader) mbar_arrive_expect_tx(&sh.bfull, (uint32_t)(kchunks * a.nq_pad * 128));
            const uint32_t bb = cluster_map(&sh.bfull, 0);
            for (int kc = 0; kc < kchunks; ++kc)
                tc::tma_load_2d_pair(bsm + (size_t)kc * bhalf * 128, &tmB, kc * 64,
                                     (int)crank * bhalf, bb);
            int s = 0, f = 0, issued = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int it = 0; it < nmine && ok; ++it) {
                int64_t r0 = ((slot0 + it * nslots) * 2 + crank) * a.tile_stride * kRows;
                if (r0 > a.rows) r0 = a.rows;   // past the end: every row out of range
                for (int k = 0; k < boxes; ++k) {
                    if (aborted(sh) || !mbar_wait(&sh.empty[s], ph)) {
                        give_up(sh, a.status);
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&sh.full[f], kBoxBytes);
                    tc::tma_load_2d_hint(ring + (size_t)s * kBoxBytes, &tmA, k * kBox, (int)r0,
                                         &sh.full[f], pol);
                    ++issued;
                    if (++f == bars) f = 0;
                    if (++s == stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            // drain: the last copy counted on every used barrier has landed before exit
            for (int b = 0; b < bars && b < issued; ++b) {
                const int last = issued - 1 - ((issued - 1 - b) % bars);
                if (!mbar_wait(&sh.full[b], turn_parity(last, stages))) give_up(sh, a.status);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (even CTA) ----------------
        // The whole warp runs the loop (uniform control flow keeps the
        // descriptors in uniform registers); one elected lane issues.
        if (leader && nmine > 0) {
            const uint32_t idesc = tc::idesc_f16_f32(2 * kRows, a.nq_pad);
            const uint64_t bd0 = tc::smem_desc_sw128_kmajor(smem_u32(bsm));
            const uint32_t bstep = (uint32_t)(bhalf * 128) >> 4;   // B, from one 64-code chunk to the next
            const bool one = tc::elect_one();
            bool ok = __all_sync(0xffffffffu, mbar_wait(&sh.bfull, 0));
            uint32_t b = 0, par = 0;
            for (int it = 0; it < nmine && ok; ++it) {
                const int acc = it & 1;
                ok = __all_sync(0xffffffffu,
                                !aborted(sh) && mbar_wait(&sh.tempty[acc],
                                                          ((uint32_t)(it >> 1) & 1u) ^ 1u));
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t d = tmem + (uint32_t)(acc * kAccCols);
                uint64_t bd = bd0;
                for (int k = 0; k < 2 * boxes; ++k) {   // half boxes of 64 codes
                    ok = __all_sync(0xffffffffu, mbar_wait(&sh.afull[b], par));
                    if (!ok) break;
                    tc::fence_after_sync();
                    if (one) {
                        if (k < kchunks) {   // (past the row's end: an empty half)
                            const uint32_t at = tmem_a + b * (uint32_t)kABufCols;
                            tc::mma_f16_pair_ts(d, at, bd, idesc, k != 0 ? 1u : 0u);
                            tc::mma_f16_pair_ts(d, at + 8, bd + 2, idesc, 1u);
                            tc::mma_f16_pair_ts(d, at + 16, bd + 4, idesc, 1u);
                            tc::mma_f16_pair_ts(d, at + 24, bd + 6, idesc, 1u);
                        }
                        tc::commit_pair(&sh.aempty[b]);
                    }
                    __syncwarp();
                    bd += bstep;
                    if (++b == kABufs) {
                        b = 0;
                        par ^= 1u;
                    }
                }
                if (ok && one) tc::commit_pair(&sh.tfull[acc]);
                __syncwarp();
            }
            if (!ok && lane == 0) give_up(sh, a.status);
            if (one) tc::commit_pair(&sh.drained);
            __syncwarp();
        }
        // every MMA issued has completed before TMEM is released
        if (nmine > 0 && !mbar_wait(&sh.drained, 0) && lane == 0) give_up(sh, a.status);
        __syncwarp();
    } else if (warp < 2 + kConvWarps) {
        // ---------------- converters ----------------
        const int grp = (warp - 2) >> 2;            // boxes g = grp, grp + 2, ...
        const int quarter = warp & 3;               // TMEM lanes this warp may write
        const int r = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const int total = nmine * boxes;
        int fb = grp;                               // the box's full barrier, and its phase
        uint32_t ph = 0;
        uint32_t b = 2 * (uint32_t)grp, aph = 1;    // the box's first half buffer, and its phase
        for (int g = grp; g < total; g += 2) {
            const int s = turn_buffer(fb, stages);
            // warp-uniform: the TMEM stores below are warp-wide
            if (!__all_sync(0xffffffffu, !aborted(sh) && mbar_wait(&sh.full[fb], ph))) {
                if (lane == 0) give_up(sh, a.status);
                break;
            }
            const uint8_t* row = ring + (size_t)s * kBoxBytes + (size_t)r * kBox;
            uint4 w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                w[c] = *reinterpret_cast<const uint4*>(row + ((c ^ (r & 7)) << 4));
            bool ok = true;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t f[32];
#pragma unroll
                for (int c = 0; c < 4; ++c) widen16(w[4 * h + c], &f[8 * c]);
                ok = ok && __all_sync(0xffffffffu, mbar_wait(&sh.aempty[b + h], aph));
                if (!ok) break;
                tc::fence_after_sync();
                tc::st_32x32b_x32(tmem_a + lane_addr + (b + h) * (uint32_t)kABufCols, f);
                tc::wait_st();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive_remote(cluster_map(&sh.afull[b + h], 0));
                    if (h == 0) mbar_arrive(&sh.empty[s]);   // the box is in registers
                }
            }
            if (!ok) {
                if (lane == 0) give_up(sh, a.status);
                break;
            }
            b ^= 4u;                                // boxes g and g + 2: the other four buffers
            if (((g >> 1) & 1) != 0) aph ^= 1u;     // both visited once
            fb += 2;
            if (fb >= bars) {
                fb -= bars;
                ph ^= 1u;
            }
        }
    } else {
        // ---------------- epilogue ----------------
        const int quarter = warp & 3;
        const int cgroup = (warp - 2 - kConvWarps) >> 2;
        const int r_in_tile = quarter * 32 + lane;
        const uint32_t lanemask_lt = (1u << lane) - 1u;
        uint2* rec = sh.rec[warp - 2 - kConvWarps];
        int nrec = 0;                               // the same in every lane
        // the last n <= 32 records, one per lane: interval, count, place
        auto settle = [&](int n) {
            nrec -= n;
            if (lane < n) {
                const uint2 e = rec[nrec + lane];
                const int64_t rw = e.x;
                const int q = (int)(e.y >> 25);
                const int dot = (int)(e.y << 7) >> 7;
                float lo, hi;
                interval_epilogue(dot, sh.qs[q], __ldg(a.scale + rw), __ldg(a.vnorm + rw),
                                  __ldg(a.enorm + rw), lo, hi);
                if (!isfinite(lo) || !isfinite(hi)) set_status(a.status, PVS_ERR_OVERFLOW);
                if (!(hi < sh.tau[q])) {
                    if (lo >= sh.tau[q]) atomicAdd(&a.h_eff[q], 1u);
                    const unsigned int pos = atomicAdd(&a.w_len[q], 1u);
                    if (pos < (unsigned int)a.w_cap) {
                        const int64_t o = (int64_t)q * a.w_cap + pos;
                        a.w_id[o] = (int32_t)rw;
                        a.w_lo[o] = lo;
                        a.w_hi[o] = hi;
                    }
                }
            }
            __syncwarp();
        };
        const uint32_t tempty_at[2] = {cluster_map(&sh.tempty[0], 0), cluster_map(&sh.tempty[1], 0)};
        // this thread's row parameters and deletion bit, loaded one tile slot
        // ahead (the norm bounds only where every row's interval is evaluated)
        float sv = 0.0f, vn = 0.0f, en = 0.0f;
        bool live = false;
        auto fetch = [&](int it, float& psv, float& pvn, float& pen, bool& plive) {
            const int64_t i = (slot0 + it * nslots) * 2 + crank;
            const int64_t rw = i * a.tile_stride * kRows + r_in_tile;
            plive = it < nmine && i < niter && rw < a.rows;
            psv = pvn = pen = 0.0f;
            if (plive) {
                psv = __ldg(a.scale + rw);
                if (a.mode == 0) {
                    pvn = __ldg(a.vnorm + rw);
                    pen = __ldg(a.enorm + rw);
                }
                plive = !tombstoned(a.tomb, rw);
            }
        };
        fetch(0, sv, vn, en, live);
        for (int it = 0; it < nmine; ++it) {
            float nsv, nvn, nen;
            bool nlive;
            fetch(it + 1, nsv, nvn, nen, nlive);
            const int64_t i = (slot0 + it * nslots) * 2 + crank;
            const int acc = it & 1;
            const bool ok = !aborted(sh) && mbar_wait(&sh.tfull[acc], (uint32_t)(it >> 1) & 1u);
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0) give_up(sh, a.status);
                break;
            }
            tc::fence_after_sync();
            const int64_t row = i * a.tile_stride * kRows + r_in_tile;
            const uint32_t tcol = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * kAccCols);
            for (int cc = cgroup; i < niter && cc < a.nq_pad / 32; cc += kEpiWarps / 4) {
                uint32_t d[32];
                tc::ld_32x32b_x32(tcol + (uint32_t)(cc * 32), d);
                tc::wait_ld();
                if (a.mode == 0 && a.group_max) {
                    // per query the row of the largest centre (of equal ones to
                    // 18 bits, the last lane's), whose own lower bound the 32
                    // rows leave; then a query in every lane.  (Every row's
                    // bound made the epilogue's instructions the sample's
                    // time: 553k x 768 x 128 queries 190 us, 113 so.)
                    int m[32];
#pragma unroll
                    for (int k = 0; k < 32; ++k) {   // (branch-free: the 32 chains overlap)
                        const float c = live ? __fmul_rn(__uint_as_float(d[k]), sv) : -INFINITY;
                        int b = __float_as_int(c);
                        b ^= (b >> 31) & 0x7fffffff;   // ordered as the floats are
                        m[k] = __reduce_max_sync(0xffffffffu, (b & ~31) | lane);
                    }
                    int best = 0;
                    uint32_t dot = 0;
#pragma unroll
                    for (int k = 0; k < 32; ++k) {
                        const uint32_t dk = __shfl_sync(0xffffffffu, d[k], m[k] & 31);
                        best = lane == k ? m[k] & 31 : best;
                        dot = lane == k ? dk : dot;
                    }
                    const float bs = __shfl_sync(0xffffffffu, sv, best);
                    const float bv = __shfl_sync(0xffffffffu, vn, best);
                    const float be = __shfl_sync(0xffffffffu, en, best);
                    const unsigned int alive = __ballot_sync(0xffffffffu, live);
                    if (cc * 32 + lane < a.nq) {
                        float lo, hi;
                        interval_epilogue(__float2int_rn(__uint_as_float(dot)),
                                          sh.qs[cc * 32 + lane], bs, bv, be, lo, hi);
                        const bool any = (alive >> best) & 1u;
                        if (any && !(isfinite(lo) && isfinite(hi)))
                            set_status(a.status, PVS_ERR_OVERFLOW);
                        a.dump_lo[(int64_t)(cc * 32 + lane) * a.dump_ld + i * 4 + quarter] =
                            any ? lo : -INFINITY;
                    }
                    continue;
                }
                if constexpr (kBounds) {
                    const int64_t at = i * kRows + r_in_tile;
#pragma unroll 1
                    for (int k = cc * 32; k < a.nq && k < cc * 32 + 32; ++k) {
                        const uint32_t v = tc::ld_32x32b_x1(tcol + (uint32_t)k);
                        tc::wait_ld();
                        float lo, hi;
                        interval_epilogue(__float2int_rn(__uint_as_float(v)), sh.qs[k], sv, vn, en,
                                          lo, hi);
                        if (live && !(isfinite(lo) && isfinite(hi)))
                            set_status(a.status, PVS_ERR_OVERFLOW);
                        a.dump_lo[(int64_t)k * a.dump_ld + at] = live ? lo : -INFINITY;
                        a.dump_hi[(int64_t)k * a.dump_ld + at] = live ? hi : -INFINITY;
                    }
                    continue;
                }
                if (a.mode == 0) {
                    const int64_t srow = i * kRows + r_in_tile;
                    bool bad = false;
#pragma unroll
                    for (int k = 0; k < 32; ++k) {   // (branch-free: the 32 chains overlap)
                        float lo, hi;
                        interval_epilogue(__float2int_rn(__uint_as_float(d[k])), sh.qs[cc * 32 + k],
                                          sv, vn, en, lo, hi);
                        bad |= live && !(isfinite(lo) && isfinite(hi));   // (padding queries: 0)
                        d[k] = __float_as_uint(live ? lo : -INFINITY);
                    }
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        if (cc * 32 + k < a.nq)
                            a.dump_lo[(int64_t)(cc * 32 + k) * a.dump_ld + srow] =
                                __uint_as_float(d[k]);
                    if (bad) set_status(a.status, PVS_ERR_OVERFLOW);
                    continue;
                }
                // any pair of the chunk that may reach its threshold?  One
                // maximum per eight queries
                const uint64_t sv2 = f2_pack(sv, sv);
                float mx[4];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    float m = -INFINITY;
#pragma unroll
                    for (int k = 8 * o; k < 8 * o + 8; k += 4) {
                        const float4 nt = *reinterpret_cast<const float4*>(&sh.ntheta[cc * 32 + k]);
                        m = max3_of(m, f2_fma(f2_pack(__uint_as_float(d[k]), __uint_as_float(d[k + 1])),
                                            sv2, f2_pack(nt.x, nt.y)));
                        m = max3_of(m, f2_fma(f2_pack(__uint_as_float(d[k + 2]),
                                                  __uint_as_float(d[k + 3])),
                                            sv2, f2_pack(nt.z, nt.w)));
                    }
                    mx[o] = live ? m : -INFINITY;   // (the maximum passes over a NaN: none here,
                }                                   //  dot and s_v are finite)
                if (!__any_sync(0xffffffffu, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) >= 0.0f))
                    continue;
                // the survivors, eight queries at a time; a group with more
                // than 32 of them is left to the loop below
                uint32_t crowded = 0;
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    if (!__any_sync(0xffffffffu, mx[o] >= 0.0f)) continue;
                    uint32_t cand = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        cand |= (uint32_t)(__fmaf_rn(__uint_as_float(d[8 * o + k]), sv,
                                                     sh.ntheta[cc * 32 + 8 * o + k]) >= 0.0f) << k;
                    if (!live) cand = 0;
                    const int mine = __popc(cand);
                    int before = __popc(__ballot_sync(0xffffffffu, mine > 0) & lanemask_lt);
                    int total = __popc(__ballot_sync(0xffffffffu, mine > 0));
                    if (__any_sync(0xffffffffu, mine > 1)) {
                        total = __reduce_add_sync(0xffffffffu, mine);
                        before = mine;   // inclusive, then exclusive prefix sum
#pragma unroll
                        for (int s = 1; s < 32; s <<= 1) {
                            const int up = __shfl_up_sync(0xffffffffu, before, s);
                            if (lane >= s) before += up;
                        }
                        before -= mine;
                    }
                    if (total > 32) {
                        crowded |= cand << (8 * o);
                        continue;
                    }
                    int at = nrec + before;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if ((cand >> k) & 1u)
                            rec[at++] = make_uint2(
                                (uint32_t)row,
                                ((uint32_t)(cc * 32 + 8 * o + k) << 25) |
                                    ((uint32_t)__float2int_rn(__uint_as_float(d[8 * o + k])) &
                                     0x1ffffffu));
                    nrec += total;
                }
                __syncwarp();
#pragma unroll 1
                while (nrec >= 32) settle(32);   // (31 + 4 x 32 records fit)
                uint32_t rest = __reduce_or_sync(0xffffffffu, crowded);
#pragma unroll 1
                while (rest != 0) {   // one column at a time, its dot products read again
                    const int k = __ffs(rest) - 1;
                    rest &= rest - 1u;
                    const uint32_t v = tc::ld_32x32b_x1(tcol + (uint32_t)(cc * 32 + k));
                    tc::wait_ld();
                    const bool take = (crowded >> k) & 1u;
                    const uint32_t who = __ballot_sync(0xffffffffu, take);
                    if (take)
                        rec[nrec + __popc(who & lanemask_lt)] = make_uint2(
                            (uint32_t)row, ((uint32_t)(cc * 32 + k) << 25) |
                                               ((uint32_t)__float2int_rn(__uint_as_float(v)) &
                                                0x1ffffffu));
                    nrec += __popc(who);
                    __syncwarp();
                    if (nrec >= 32) settle(32);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(tempty_at[acc]);
            sv = nsv;
            vn = nvn;
            en = nen;
            live = nlive;
        }
        settle(nrec);
    }
    __syncthreads();
    cluster_barrier();   // no CTA leaves while its peer may still address it
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc_pair(tmem, kTmemCols);
    }
}

// theta_q such that dot * s_v < theta_q implies hi < tau_q for every row.
// hi = RU(c + r) with r <= rmax_q (each factor of App. A.1's half-width at its
// corpus maximum, |c| at most cmax; all operations rounded up and monotone),
// and c = RN(RN(s_q s_v) dot) is within cmax 2^-22 (and 2^-140 where it
// underflows) of s_q (s_v dot).  So s_q (dot s_v) <= tau' - rmax_q - slack
// suffices, with tau' below tau's float32 predecessor.  In binary64 (errors
// far inside the slack); one thread per query.
__global__ void stream_theta_kernel(const QueryScalars* qs, int nq, const unsigned int* maxes,
                                    const float* tau, float* theta) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    const QueryScalars s = qs[q];
    const float vmax = __uint_as_float(maxes[0]), emax = __uint_as_float(maxes[1]);
    const float E = __fadd_ru(__fmul_ru(s.enorm, vmax), __fmul_ru(s.qhat, emax));
    const float cmax = __fmul_ru(__fmul_ru(s.qhat, __fadd_ru(vmax, emax)), 1.0f + 0x1p-21f);
    const float G = __fmul_ru(__fadd_ru(__fadd_ru(cmax, E), __fmul_ru(s.qnorm, vmax)), s.gamma);
    const double rmax = (double)__fadd_ru(E, G);
    const double t = (double)tau[q];
    const double need = t - fabs(t) * 0x1p-22 - rmax - (double)cmax * 0x1p-21 - 0x1p-130;
    const float th = __double2float_rd(need / (double)s.s);
    theta[q] = th == th ? th : -INFINITY;   // (a NaN rejects nothing)
}

size_t fixed_smem(int m_pad, int nq_pad) {
    return 1024 + (size_t)(m_pad / 64) * (nq_pad / 2) * 128 + sizeof(StreamShared);
}
int stream_stages(int m_pad, int nq_pad) {
    const size_t fixed = fixed_smem(m_pad, nq_pad);
    if (fixed + 2 * kBoxBytes > (size_t)kSmemMax) return 0;
    const int s = (int)(((size_t)kSmemMax - fixed) / kBoxBytes);
    return s < kMaxStages ? s : kMaxStages;
}

cudaLaunchConfig_t stream_config(int grid, size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kStreamThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    return cfg;
}

// CTA pairs of the kernel that run at once on the current device (0: none).
int stream_pairs(int num_sms) {
    static std::mutex mu;
    static int pairs[64];
    static bool known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 0;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!known[dev]) {
        int n = 0;
        if (raise_smem_limit((const void*)batch_stream_kernel<false>, kSmemMax) == cudaSuccess) {
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 2;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = stream_config(2 * num_sms, kSmemMax, nullptr);
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, batch_stream_kernel<false>, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
        } else {
            cudaGetLastError();
        }
        pairs[dev] = n;
        known[dev] = true;
    }
    return pairs[dev];
}

}  // namespace

// Queries of one pass: as many as leave four boxes of the ring (98 KB of B).
int batch_stream_queries(int m_pad) {
    const int q = (96 * 1024) / m_pad / 32 * 32;   // m_pad f16 per query, half of them per CTA
    return q < kStreamQueries ? q : kStreamQueries;
}

bool batch_stream_supported(int m_pad, int num_sms) {
    return m_pad >= kBox && m_pad <= kStreamMaxWidth && m_pad % 64 == 0 && stream_pairs(num_sms) > 0;
}

cudaError_t launch_stream_theta(const QueryScalars* qs, int nq, const unsigned int* maxes,
                                const float* tau, float* theta, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    count_launches(1);
    stream_theta_kernel<<<(nq + 31) / 32, 32, 0, st>>>(qs, nq, maxes, tau, theta);
    return cudaGetLastError();
}

cudaError_t launch_batch_stream(const StreamArgs& a, const int8_t* codes, const uint16_t* qcodes,
                                int num_sms, cudaStream_t st) {
    if (a.rows <= 0 || a.nq <= 0) return cudaSuccess;
    if (a.nq > kStreamQueries || a.nq_pad % 32 != 0 || a.nq_pad < a.nq ||
        a.nq_pad > kStreamQueries || a.tile_stride < 1 || a.rows >= ((int64_t)1 << 31) ||
        !batch_stream_supported(a.m_pad, num_sms))
        return cudaErrorInvalidValue;
    const int stages = stream_stages(a.m_pad, a.nq_pad);
    if (stages < 2) return cudaErrorInvalidValue;
    CUtensorMap ta, tb;
    if (!tensor_map_2d(&ta, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, codes, (uint64_t)a.rows,
                    (uint64_t)a.m_pad, kBox, kRows) ||
        !tensor_map_2d(&tb, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, qcodes, (uint64_t)a.nq_pad,
                    (uint64_t)a.m_pad, 64, (uint32_t)(a.nq_pad / 2)))
        return cudaErrorInvalidValue;
    const int64_t ntiles = (a.rows + kRows - 1) / kRows;
    const int64_t niter = (ntiles + a.tile_stride - 1) / a.tile_stride;
    const int64_t slots = (niter + 1) / 2;
    const int pairs = stream_pairs(num_sms);
    const int grid = 2 * (int)(slots < pairs ? slots : pairs);
    const size_t smem = fixed_smem(a.m_pad, a.nq_pad) + (size_t)stages * kBoxBytes;
    auto run = [&](auto kernel) {
        const cudaError_t e = raise_smem_limit((const void*)kernel, kSmemMax);
        if (e != cudaSuccess) return e;
        count_launches(1);
        kernel<<<grid, kStreamThreads, smem, st>>>(ta, tb, a, stages);
        return cudaGetLastError();
    };
    return a.dump_hi ? run(batch_stream_kernel<true>) : run(batch_stream_kernel<false>);
}

// f16 copy of int8 codes (exact: |z| <= 127); rows past n become zeros.
__global__ void codes_to_f16_kernel(const int8_t* __restrict__ src, uint16_t* __restrict__ dst,
                                    int64_t count, int64_t padded) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= padded) return;
    uint16_t h = 0;
    if (i < count) asm("cvt.rn.f16.s16 %0, %1;" : "=h"(h) : "h"((short)src[i]));
    dst[i] = h;
}

cudaError_t launch_codes_to_f16(const int8_t* src, uint16_t* dst, int64_t count, int64_t padded,
                                cudaStream_t st) {
    if (padded <= 0) return cudaSuccess;
    count_launches(1);
    codes_to_f16_kernel<<<(unsigned)((padded + 255) / 256), 256, 0, st>>>(src, dst, count, padded);
    return cudaGetLastError();
}

}  // namespace pvs
