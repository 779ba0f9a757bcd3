// PVS index build and query encoding (Sec. 2.3.1; norms for App. A.1).
//
// One warp quantizes one vector: float32 loads, warp max of |v_j|, the scale
// by IEEE division, the codes, and the order-independent integer
// accumulation of the norm bounds (the arithmetic quantize_row_warp states).
// The raw float32 row is copied next to the codes for authoritative scoring.
#include <algorithm>

#include "f32x2.cuh"
#include "kernels.h"
#include "pipeline.cuh"
#include "pvs_common.cuh"

namespace pvs {

// Rows the integer arithmetic below does not cover (all-subnormal rows or
// residuals, scales under 2^-100, a residual past the float32 grid): the
// binary64 quantizer.  Out of line: never taken on ordinary data.
static __device__ __noinline__ RowQuant quantize_row_slow(const float* v, int m, int m_pad, int8_t* z,
                                                   float fixed_s) {
    return quantize_row_warp(v, m, m_pad, z, fixed_s);
}

// A sum of squares x^2 2^(-2e), |x| < 2^e, to about 2^-37 of its value, two
// chains of float32 at a time: s from 1 on, so that it is at least each
// product and s' = RN(s + p) has the exact error p - (s' - s) (Dekker's
// FastTwoSum); the products' errors are exact too (one FMA), and both sum to c.
// n squares a chain: |c| <= 2 n u s with u = 2^-24, and the 2 n additions to it
// and that of two chains' c round by u |c| at most, so 64 chains err by at most
// 4 n (n + 1) u^2 (64 + S) in all.
struct SquareSum {
    uint64_t s, c = 0;
    const uint64_t scale, neg_scale, m1;   // 2^-e, -2^-e, -1 in both halves
    __device__ __forceinline__ explicit SquareSum(float f)
        : s(f2_pack(1.0f, 1.0f)), scale(f2_pack(f, f)), neg_scale(f2_pack(-f, -f)),
          m1(f2_pack(-1.0f, -1.0f)) {}
    __device__ __forceinline__ void add(float a, float b) {
        const uint64_t v = f2_pack(a, b);
        const uint64_t x = f2_mul(v, scale);
        const uint64_t np = f2_mul(x, f2_mul(v, neg_scale));   // -RN(x^2)
        const uint64_t ep = f2_fma(x, x, np);
        const uint64_t s1 = f2_fma(np, m1, s);                 // s + p
        const uint64_t es = f2_fma(np, m1, f2_fma(s1, m1, s));
        c = f2_add(c, f2_add(ep, es));
        s = s1;
    }
    // The sum over the warp's 64 chains in units of 2^-38 (the same in every
    // lane): s - 1 is a multiple of 2^-23, below 2^5 for up to 32 squares a lane;
    // c rounds by half a unit a lane.
    __device__ __forceinline__ long long warp_total() const {
        float s0, s1, c0, c1;
        f2_unpack(s, s0, s1);
        f2_unpack(c, c0, c1);
        const int a = (int)__fmul_rn(__fsub_rn(s0, 1.0f), 0x1p23f) +
                      (int)__fmul_rn(__fsub_rn(s1, 1.0f), 0x1p23f);
        const int b = __float2int_rn(__fmul_rn(__fadd_rn(c0, c1), 0x1p38f));
        const int ahi = __reduce_add_sync(0xffffffffu, a >> 16);
        const int alo = __reduce_add_sync(0xffffffffu, a & 0xffff);
        const int bt = __reduce_add_sync(0xffffffffu, b);
        return ((((long long)ahi << 16) + alo) << 15) + bt;
    }
};
// 2^-e for the biased exponent field E of the largest |x| (e = E - 126)
__device__ __forceinline__ float norm_scale(int E) {
    return E <= 252 ? __uint_as_float((uint32_t)(253 - E) << 23) : __uint_as_float(0x00400000u >> (E - 253));
}
// norm_finish of the integer sum T of norm_term_bits, from the total of a
// SquareSum of n squares a chain, of m in all: T 2^-48 lies in [S, S + m 2^-48).
// Both ends of the interval round to the same bound, or *settled is false.
__device__ inline float norm_from_squares(long long total, int e, int n, int m, bool* settled) {
    const double S = (double)total * 0x1p-38;
    const double u2 = 4.04 * 0x1p-48 * (double)(n * (n + 1));
    const double E = u2 * (64.0 + S) + 0x1p-33 + (double)m * 0x1p-48;
    const double r = __dsqrt_rn(S) * pow2d(e);
    // |sqrt(S + d) / sqrt(S) - 1| <= |d| / S for |d| <= S / 2
    const double d = r * (E / S + 0x1p-50);
    const float lo = __double2float_ru(r - d), hi = __double2float_ru(r + d);
    *settled = lo == hi;
    return hi;
}
// Both integer sums of a row again, exactly, by the warp: the rows whose
// intervals hold a rounding boundary (one norm in about 2^12).
static __device__ __noinline__ void exact_norm_sums(const float* v, int m, float s, int Ev, int Ee,
                                                    unsigned long long* T) {
    const float rs = __frcp_rn(s);
    unsigned long long a = 0, b = 0;
    for (int j = threadIdx.x & 31; j < m; j += kWarp) {
        uint32_t y;
        const float x = v[j];
        const float e = __fmaf_rn(-s, code_of(x, s, rs, y), x);
        a += norm_term_bits(__float_as_uint(fabsf(x)), Ev);
        b += norm_term_bits(__float_as_uint(fabsf(e)), Ee);
    }
    T[0] = warp_sum(a);
    T[1] = warp_sum(b);
}

// One warp per row, `per_warp` (<= 32) rows of a warp in turn.  Everything per
// element is float32 and integer work:
//   - the code comes from the product with 1 / s (code_of);
//   - the residual v - s c is exact in one FMA: v and s c are multiples of
//     u = max(ulp(s) / 2, 2^-149) (v >= s / 2 where c != 0) and
//     |v - s c| < 2^floor(log2 s) <= 2^24 u, checked per row;
//   - the norm bounds are those of sums of norm_term_bits, found from a sum of
//     squares with an error bound (SquareSum); wider rows sum the terms.
// Lane r keeps the sums of the batch's r-th row, and the binary64 square
// roots run once for the batch, one row per lane.
//
// Bound by: HBM (4m bytes read, 5m + 12 written per row); the element work is
// about 25 instructions.  With binary64 norm terms and four passes over the row
// the FP64 pipe was the bound (500k x 768: 12.1 ms), then the latency of
// one row after the other (1,290 us with integer terms, 1,166 with sums of
// squares): a warp's loads waited for its last row's reductions.  Rows now come
// ahead through a ring of bulk copies, two or three per warp: 628 us
// (5.5 TB/s), 1M x 1,024 3,670 -> 1,606 us, 1M x 384 1,048 -> 693 us, 2M x 128
// 867 -> 797 us.  Three
// blocks of fewer registers from 513 dimensions on: 670 and 1,920 us.
// NV4: float4 of the row per lane, in registers (m_pad <= 128 NV4); 0: wider
// rows are read again (from L1 / L2) in each of the three steps.

template <int NV4>
__global__ void __launch_bounds__(256, NV4 > 4 ? 2 : 4) build_kernel(const float* __restrict__ vecs, int64_t n,
                                                    int m, int m_pad, int m_raw,
                                                    int8_t* __restrict__ codes,
                                                    float* __restrict__ scale,
                                                    float* __restrict__ vnorm,
                                                    float* __restrict__ enorm,
                                                    float* __restrict__ raw, int* status,
                                                    const float* fixed_scale, int aligned,
                                                    int per_warp, int stages) {
    constexpr int kKeep = NV4 > 0 ? NV4 : 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t stride = (int64_t)gridDim.x * (blockDim.x >> 5) * per_warp;
    const float fs = fixed_scale ? *fixed_scale : 0.0f;
    const int steps = NV4 > 0 ? NV4 : (m_pad + 127) / 128;
    const int64_t first = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * per_warp;
    // the ring: rows [warps][stages][m] | barriers [warps][stages]; lane 0
    // issues the rows in the order they are read
    extern __shared__ float4 build_ring[];
    const int n4 = m >> 2;
    float4* ring = build_ring + (size_t)warp * stages * n4;
    uint64_t* bars = reinterpret_cast<uint64_t*>(build_ring + (size_t)(blockDim.x >> 5) * stages * n4) +
                     warp * stages;
    const uint32_t row_bytes = (uint32_t)m * sizeof(float);
    uint64_t pol = 0;
    int64_t next0 = first;   // the next row to issue: next0 + nextb
    int nextb = 0;
    int in_flight = 0;       // rows issued and not read; the oldest in buffer st
    int st = 0;
    uint32_t parity = 0;     // of buffer st
    auto issue = [&](int buf) {
        if (next0 >= n) return;
        if (lane == 0) {
            fence_proxy_async_smem();   // the warp's reads of this buffer come first
            mbar_arrive_expect_tx(&bars[buf], row_bytes);
            bulk_g2s(ring + (size_t)buf * n4, vecs + (next0 + nextb) * (int64_t)m, row_bytes,
                     &bars[buf], pol);
        }
        ++in_flight;
        if (++nextb == per_warp || next0 + nextb >= n) {
            nextb = 0;
            next0 += stride;
        }
    };
    if (NV4 > 0 && stages) {
        if (lane == 0) {
            pol = l2_evict_first_policy();
            for (int b = 0; b < stages; ++b) mbar_init(&bars[b], 1);
            mbar_fence_init();
        }
        __syncwarp();
        for (int b = 0; b < stages; ++b) issue(b);
    }
    for (int64_t row0 = first; row0 < n; row0 += stride) {
        const int batch = (int)(n - row0 < per_warp ? n - row0 : per_warp);
        // this lane's row of the batch
        unsigned long long tv = 0, te = 0;
        int ev = 0, ee = 0;
        float s_of = 0.0f, vn = 0.0f, en = 0.0f;
        bool done = false;
        for (int b = 0; b < batch; ++b) {
            const int64_t row = row0 + b;
            const float* v = vecs + row * (int64_t)m;
            auto load = [&](int i) {
                const int j = 4 * (lane + 32 * i);
                float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (NV4 > 0 && stages) {
                    if (j < m) x = ring[(size_t)st * n4 + (j >> 2)];
                } else if (aligned) {
                    if (j < m) x = __ldcs(reinterpret_cast<const float4*>(v + j));
                } else {
                    if (j < m) x.x = v[j];
                    if (j + 1 < m) x.y = v[j + 1];
                    if (j + 2 < m) x.z = v[j + 2];
                    if (j + 3 < m) x.w = v[j + 3];
                }
                return x;
            };
            float4 keep[kKeep];
            uint32_t mx = 0;
            // warp-uniform: every lane must agree before the warp-wide steps below
            if (NV4 > 0 && stages && !__all_sync(0xffffffffu, mbar_wait(&bars[st], parity))) {
                // a copy did not arrive in time: record it, drain every copy in flight
                if (lane == 0) set_status(status, PVS_ERR_TIMEOUT);
                for (int k = 0; k < in_flight; ++k) {
                    mbar_wait(&bars[st], parity);
                    if (++st == stages) st = 0, parity ^= 1u;
                }
                return;
            }
#pragma unroll
            for (int i = 0; i < steps; ++i) {
                const float4 x = load(i);
                if constexpr (NV4 > 0) keep[i] = x;
                const int j = 4 * (lane + 32 * i);
                if (j < m_raw) *reinterpret_cast<float4*>(raw + row * (int64_t)m_raw + j) = x;
                mx = max(max(mx, __float_as_uint(fabsf(x.x))), __float_as_uint(fabsf(x.y)));
                mx = max(max(mx, __float_as_uint(fabsf(x.z))), __float_as_uint(fabsf(x.w)));
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            if (NV4 > 0 && stages) {   // every lane has its values: the buffer is free
                --in_flight;
                issue(st);
                if (++st == stages) st = 0, parity ^= 1u;
            }
            if (mx >= 0x7f800000u) {   // an infinity or a NaN
                if (lane == 0) set_status(status, PVS_ERR_NONFINITE);
                done |= lane == b;
                continue;
            }
            float s = fs;
            if (!(fs > 0.0f)) s = mx == 0 ? 1.0f : __fdiv_rn(__uint_as_float(mx), 127.0f);
            const float rs = __frcp_rn(s);
            uint32_t emx = 0;
            bool out_of_range = false;
            uint32_t* zrow = reinterpret_cast<uint32_t*>(codes + row * (int64_t)m_pad);
            bool slow = mx != 0 && (mx < 0x00800000u || s < kFastScaleMin);
            const int Ev = max((int)(mx >> 23), 1);   // (0: sums of 0)
            unsigned long long a = 0, c2 = 0;
            SquareSum sq(NV4 > 0 ? norm_scale(Ev) : 0.0f);
            if (!slow) {
#pragma unroll
                for (int i = 0; i < steps; ++i) {
                    const float4 x = NV4 > 0 ? keep[NV4 > 0 ? i : 0] : load(i);
                    uint32_t y[4];
                    const float xs[4] = {x.x, x.y, x.z, x.w};
                    float e[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float c = code_of(xs[k], s, rs, y[k]);
                        if (fs > 0.0f && fabsf(c) > 127.0f) out_of_range = true;
                        e[k] = __fmaf_rn(-s, c, xs[k]);
                        emx = max(emx, __float_as_uint(fabsf(e[k])));
                        if constexpr (NV4 == 0) a += norm_term_bits(__float_as_uint(fabsf(xs[k])), Ev);
                    }
                    if constexpr (NV4 > 0) {
                        sq.add(x.x, x.y);
                        sq.add(x.z, x.w);
                    }
                    const int j4 = lane + 32 * i;
                    if (4 * j4 < m_pad)
                        zrow[j4] = __byte_perm(__byte_perm(y[0], y[1], 0x0040),
                                               __byte_perm(y[2], y[3], 0x0040), 0x5410);
                    if constexpr (NV4 > 0) keep[i] = make_float4(e[0], e[1], e[2], e[3]);
                }
                emx = __reduce_max_sync(0xffffffffu, emx);
                // not on the residual's float32 grid, or a subnormal maximum
                slow = emx >= (__float_as_uint(s) & 0x7f800000u) || (emx != 0 && emx < 0x00800000u);
                if (fs > 0.0f && __any_sync(0xffffffffu, out_of_range)) slow = true;
            }
            if (slow) {   // the same for the whole warp
                __syncwarp();
                const RowQuant r =
                    quantize_row_slow(v, m, m_pad, codes + row * (int64_t)m_pad, fs);
                if (lane == b) {
                    s_of = r.s;
                    vn = r.vnorm;
                    en = r.enorm;
                    done = true;
                }
                if (r.status && lane == 0) set_status(status, r.status);
                continue;
            }
            const int Ee = max((int)(emx >> 23), 1);
            SquareSum eq(NV4 > 0 ? norm_scale(Ee) : 0.0f);
#pragma unroll
            for (int i = 0; i < steps; ++i) {
                if constexpr (NV4 > 0) {
                    eq.add(keep[i].x, keep[i].y);
                    eq.add(keep[i].z, keep[i].w);
                } else {
                    const float4 x = load(i);
                    const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t y;
                        const float e = __fmaf_rn(-s, code_of(xs[k], s, rs, y), xs[k]);
                        c2 += norm_term_bits(__float_as_uint(fabsf(e)), Ee);
                    }
                }
            }
            if constexpr (NV4 > 0) {
                a = mx ? (unsigned long long)sq.warp_total() : 0ull;
                c2 = emx ? (unsigned long long)eq.warp_total() : 0ull;
            } else {
                a = warp_sum(a);
                c2 = warp_sum(c2);
            }
            if (lane == b) {
                s_of = s;
                tv = a;
                te = c2;
                ev = Ev - 126;
                ee = Ee - 126;
            }
        }
        if constexpr (NV4 > 0) {
            bool open = false;
            if (lane < batch && !done) {
                bool ok = true;
                vn = tv ? norm_from_squares((long long)tv, ev, 2 * NV4, m, &ok) : 0.0f;
                open = !ok;
                en = te ? norm_from_squares((long long)te, ee, 2 * NV4, m, &ok) : 0.0f;
                open |= !ok;
            }
            unsigned int todo = __ballot_sync(0xffffffffu, open);
            while (todo) {
                const int b = __ffs(todo) - 1;
                todo &= todo - 1;
                unsigned long long T[2];
                const int Ev = __shfl_sync(0xffffffffu, ev, b) + 126;
                const int Ee = __shfl_sync(0xffffffffu, ee, b) + 126;
                exact_norm_sums(vecs + (row0 + b) * (int64_t)m, m,
                                __shfl_sync(0xffffffffu, s_of, b), Ev, Ee, T);
                if (lane == b) {
                    vn = norm_finish((long long)T[0], ev);
                    en = norm_finish((long long)T[1], ee);
                }
            }
        }
        if (lane < batch) {
            if (!done) {
                if constexpr (NV4 == 0) {
                    vn = norm_finish((long long)tv, ev);
                    en = norm_finish((long long)te, ee);
                }
                if (isinf(vn) || isinf(en)) set_status(status, PVS_ERR_OVERFLOW);
            }
            scale[row0 + lane] = s_of;
            vnorm[row0 + lane] = vn;
            enorm[row0 + lane] = en;
        }
    }
}

cudaError_t launch_build(const float* vecs, int64_t n, int m, int m_pad, int m_raw,
                         int8_t* codes, float* scale, float* vnorm, float* enorm, float* raw,
                         int* status, cudaStream_t st, const float* fixed_scale) {
    if (n <= 0) return cudaSuccess;
    // the binary64 roots cost a warp the same for 1 row or 32: long batches
    // once there are rows enough for every warp of the chip
    const int per_warp = (int)std::min<int64_t>(32, std::max<int64_t>(1, n / (152 * 32)));
    int64_t blocks = (n + 8 * per_warp - 1) / (8 * per_warp);
    if (blocks > 152 * 64) blocks = 152 * 64;
    const int aligned =
        m % 4 == 0 && (reinterpret_cast<uintptr_t>(vecs) & 15u) == 0 ? 1 : 0;
    // rows of up to 1,024 dimensions on 16-byte boundaries come through the
    // ring, three a warp where three blocks of them fit on an SM
    const size_t row = (size_t)m * sizeof(float) + sizeof(uint64_t);
    const int stages = !aligned || m_pad > 1024 ? 0 : 3 * 8 * 3 * row <= 216 * 1024 ? 3 : 2;
    const size_t smem = 8 * (size_t)stages * row;
    auto run = [&](auto kernel) {
        const cudaError_t e = raise_smem_limit((const void*)kernel, smem);
        if (e != cudaSuccess) return e;
        count_launches(1);
        kernel<<<(unsigned)blocks, 256, smem, st>>>(vecs, n, m, m_pad, m_raw, codes, scale, vnorm,
                                                    enorm, raw, status, fixed_scale, aligned,
                                                    per_warp, stages);
        return cudaGetLastError();
    };
    switch ((m_pad + 127) / 128) {
        case 1: return run(build_kernel<1>);
        case 2: return run(build_kernel<2>);
        case 3: return run(build_kernel<3>);
        case 4: return run(build_kernel<4>);
        case 5: return run(build_kernel<5>);
        case 6: return run(build_kernel<6>);
        case 7: return run(build_kernel<7>);
        case 8: return run(build_kernel<8>);
        default: return run(build_kernel<0>);
    }
}

// Largest |v_j| over count floats, as float bits (nonnegative floats order
// like their bits; a NaN entry wins and makes the scale NaN, and the build
// then reports the non-finite row).
__global__ void maxabs_kernel(const float* __restrict__ v, int64_t count, unsigned int* out) {
    unsigned int m = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride)
        m = max(m, __float_as_uint(fabsf(v[i])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// s = RN(maxabs / 127), 1 for an all-zero corpus, 2^-149 if the quotient underflows.
__global__ void scale_from_maxabs_kernel(const unsigned int* maxabs_bits, float* s) {
    const float mx = __uint_as_float(*maxabs_bits);
    float v = 1.0f;
    if (mx != 0.0f) {
        v = __fdiv_rn(mx, 127.0f);
        if (v == 0.0f) v = __uint_as_float(1u);
    }
    *s = v;
}

cudaError_t launch_maxabs(const float* v, int64_t count, unsigned int* out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    count_launches(1);
    maxabs_kernel<<<(unsigned)blocks, 256, 0, st>>>(v, count, out);
    return cudaGetLastError();
}

cudaError_t launch_scale_from_maxabs(const unsigned int* maxabs_bits, float* s, cudaStream_t st) {
    count_launches(1);
    scale_from_maxabs_kernel<<<1, 1, 0, st>>>(maxabs_bits, s);
    return cudaGetLastError();
}

// Queries: one block of kEncThreads per query, the quantizer of the rows
// spread over its warps (maxima and exact integer sums do not depend on the
// order, so the results are bit-identical), plus the query-side scalars of
// App. A.1: ||s_q z_q|| rounded up and gamma_m = RU(a / RD(1 - a)),
// a = (8m + 64) 2^-23.
// q and qraw may be the same buffer (a host query staged in qraw): the raw
// copy rewrites the values that the first loop read.
// Bound by latency (one block, a few values per thread): float32 and integer
// terms as in build_kernel, three block barriers, and the three square roots
// on three warps side by side.
constexpr int kEncThreads = 256;
constexpr int kEncWarps = kEncThreads / kWarp;

struct EncShared {
    uint32_t u[kEncWarps][2];
    unsigned long long t[kEncWarps][3];
    float root[3];
};

// The scalars of a query outside the fast path (see build_kernel), in
// binary64 by one warp; codes to z.
static __device__ __noinline__ QueryScalars encode_query_slow(const float* v, int m, int m_pad,
                                                              int8_t* z) {
    const int lane = threadIdx.x & 31;
    const RowQuant r = quantize_row_warp(v, m, m_pad, z);
    QueryScalars out{};
    out.status = r.status;
    out.s = r.s;
    out.qnorm = r.vnorm;
    out.enorm = r.enorm;
    // ||q_hat||: the values s z_j are exact in binary64
    double M = 0.0;
    for (int j = lane; j < m; j += kWarp) M = fmax(M, fabs(__dmul_rn((double)r.s, (double)z[j])));
    M = warp_max(M);
    long long T = 0;
    const int e = M > 0.0 ? norm_exponent(M) : 0;
    if (M > 0.0)
        for (int j = lane; j < m; j += kWarp) T += norm_term(__dmul_rn((double)r.s, (double)z[j]), e);
    out.qhat = norm_finish(warp_sum(T), e);
    if (out.status == 0 && isinf(out.qhat)) out.status = PVS_ERR_OVERFLOW;
    return out;
}

__global__ void __launch_bounds__(kEncThreads) encode_kernel(const float* q, int nq, int m,
                                                            int m_pad, int m_raw,
                                                            int8_t* __restrict__ zq, float* qraw,
                                                            QueryScalars* __restrict__ qs,
                                                            DevCounters* ctr, int* status,
                                                            int* status_mirror) {
    __shared__ EncShared sh;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int qi = blockIdx.x;
    if (qi >= nq) return;
    const float* v = q + (int64_t)qi * m;
    float* raw = qraw + (int64_t)qi * m_raw;
    int8_t* z = zq + (int64_t)qi * m_pad;
    constexpr int kKeep = 4;   // values per thread held in registers (1,024 dimensions)
    float keep[kKeep];
    // f(j, q_j) for this thread's j < limit (q_j = 0 from m on)
    auto each = [&](int limit, auto f) {
#pragma unroll
        for (int i = 0; i < kKeep; ++i)
            if (t + i * kEncThreads < limit) f(t + i * kEncThreads, keep[i]);
        for (int j = t + kKeep * kEncThreads; j < limit; j += kEncThreads)
            f(j, j < m ? v[j] : 0.0f);
    };
    const float a = (float)((8.0 * (double)m + 64.0) * 0x1p-23);   // exact
    const float gamma = __fdiv_ru(a, __fsub_rd(1.0f, a));
    // the thread that stores the scalars publishes them
    auto publish = [&](const QueryScalars& out) {
        qs[qi] = out;
        if (ctr) *ctr = DevCounters{};
        if (status) *status = 0;
        if (status_mirror) {
            __threadfence_system();
            *reinterpret_cast<volatile int*>(status_mirror) = out.status;
        }
    };
    // finiteness and max |q_j|
    uint32_t mx = 0;
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
        const int j = t + i * kEncThreads;
        keep[i] = j < m ? v[j] : 0.0f;
    }
    each(m_raw, [&](int j, float x) {
        mx = max(mx, __float_as_uint(fabsf(x)));
        raw[j] = x;
    });
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) sh.u[warp][0] = mx;
    __syncthreads();
    for (int w = 0; w < kEncWarps; ++w) mx = max(mx, sh.u[w][0]);
    if (mx >= 0x7f800000u) {   // an infinity or a NaN
        if (t == 0) {
            QueryScalars out{};
            out.status = PVS_ERR_NONFINITE;
            out.gamma = gamma;
            publish(out);
        }
        return;
    }
    const float s = mx == 0 ? 1.0f : __fdiv_rn(__uint_as_float(mx), 127.0f);
    bool slow = mx != 0 && (mx < 0x00800000u || s < kFastScaleMin);
    __syncthreads();   // sh.u is written again
    // codes, residual maximum, largest code
    const float rs = __frcp_rn(s);
    uint32_t emx = 0, zmx = 0;
    if (!slow) {
        each(m_pad, [&](int j, float x) {
            uint32_t y;
            const float c = code_of(x, s, rs, y);
            z[j] = (int8_t)(y & 0xffu);
            emx = max(emx, __float_as_uint(fabsf(__fmaf_rn(-s, c, x))));
            zmx = max(zmx, (uint32_t)fabsf(c));
        });
        emx = __reduce_max_sync(0xffffffffu, emx);
        zmx = __reduce_max_sync(0xffffffffu, zmx);
        if (lane == 0) {
            sh.u[warp][0] = emx;
            sh.u[warp][1] = zmx;
        }
        __syncthreads();
        for (int w = 0; w < kEncWarps; ++w) {
            emx = max(emx, sh.u[w][0]);
            zmx = max(zmx, sh.u[w][1]);
        }
        slow = emx >= (__float_as_uint(s) & 0x7f800000u) || (emx != 0 && emx < 0x00800000u);
    }
    if (slow) {
        __syncthreads();   // the codes above are rewritten
        if (warp == 0) {
            QueryScalars out = encode_query_slow(raw, m, m_pad, z);
            out.gamma = gamma;
            if (lane == 0) publish(out);
        }
        return;
    }
    // norm bounds of q, of its residual and of q_hat = s z: with s = S 2^p
    // (S < 2^24), (s z)^2 = (S |z|)^2 2^(2p), and the largest S |z| has
    // `bits` bits, so t = ceil((S |z|)^2 / 2^(2 bits - 48))
    const int Ev = max((int)(mx >> 23), 1), Ee = max((int)(emx >> 23), 1);
    const uint32_t S = (__float_as_uint(s) & 0x7fffffu) | 0x800000u;
    const int bits = 32 - __clz((int)(S * zmx));
    const int dh = max(2 * bits - 48, 0);   // (bits >= 24 unless every code is 0)
    unsigned long long T[3] = {0, 0, 0};
    each(m, [&](int, float x) {
        uint32_t y;
        const float c = code_of(x, s, rs, y);
        T[0] += norm_term_bits(__float_as_uint(fabsf(x)), Ev);
        T[1] += norm_term_bits(__float_as_uint(fabsf(__fmaf_rn(-s, c, x))), Ee);
        const unsigned long long P = (unsigned long long)S * (uint32_t)fabsf(c);
        T[2] += (P * P + ((1ull << dh) - 1ull)) >> dh;
    });
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        T[k] = warp_sum(T[k]);
        if (lane == 0) sh.t[warp][k] = T[k];
    }
    __syncthreads();
    if (lane == 0 && warp < 3) {
        unsigned long long sum = 0;
        for (int w = 0; w < kEncWarps; ++w) sum += sh.t[w][warp];
        // exponent of the maximum: M = f 2^e with f in [0.5, 1)
        const int es = (int)(__float_as_uint(s) >> 23) - 150 + bits;
        const int e = warp == 0 ? Ev - 126 : warp == 1 ? Ee - 126 : es;
        sh.root[warp] = norm_finish((long long)sum, e);
    }
    __syncthreads();
    if (t == 0) {
        QueryScalars out{};
        out.s = s;
        out.qnorm = sh.root[0];
        out.enorm = sh.root[1];
        out.qhat = sh.root[2];
        out.gamma = gamma;
        if (isinf(out.qnorm) || isinf(out.enorm) || isinf(out.qhat)) out.status = PVS_ERR_OVERFLOW;
        publish(out);
    }
}

cudaError_t launch_encode_query(const float* q, int m, int m_pad, int m_raw, int8_t* zq,
                                float* qraw, QueryScalars* qs, DevCounters* ctr, int* status,
                                int* status_mirror, cudaStream_t st) {
    count_launches(1);
    encode_kernel<<<1, kEncThreads, 0, st>>>(q, 1, m, m_pad, m_raw, zq, qraw, qs, ctr, status,
                                             status_mirror);
    return cudaGetLastError();
}

cudaError_t launch_encode_queries(const float* q, int nq, int m, int m_pad, int m_raw,
                                  int8_t* zq, float* qraw, QueryScalars* qs, cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    count_launches(1);
    encode_kernel<<<nq, kEncThreads, 0, st>>>(q, nq, m, m_pad, m_raw, zq, qraw, qs, nullptr,
                                              nullptr, nullptr);
    return cudaGetLastError();
}

}  // namespace pvs
