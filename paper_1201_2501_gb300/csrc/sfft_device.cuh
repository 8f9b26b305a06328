// sfft_device.cuh -- device helpers shared by the exact and the general kernels: complex
// arithmetic, the precision-templated transcendental helpers, block-wide scan/sort and the batched
// bin FFT.  Everything is inline; each translation unit gets its own copy.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "sfft_internal.h"

namespace sfft {

// ------------------------------------------------------------------------------------------------
// complex helpers
// ------------------------------------------------------------------------------------------------
template <typename R>
struct Cx;
template <>
struct Cx<float> {
    using T = float2;
};
template <>
struct Cx<double> {
    using T = double2;
};

__device__ __forceinline__ float2 mkc(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mkc(double a, double b) { return make_double2(a, b); }
template <typename C>
__device__ __forceinline__ C cadd(C a, C b) {
    a.x += b.x;
    a.y += b.y;
    return a;
}
template <typename C>
__device__ __forceinline__ C csub(C a, C b) {
    a.x -= b.x;
    a.y -= b.y;
    return a;
}
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
// b w with each product and sum rounded as written in any context (a compiler may otherwise merge the
// product into the sums of an unrolled FFT pass): the roundings of cmul where it is not merged
__device__ __forceinline__ float2 cmul_rn(float2 b, float2 w) {
    return make_float2(__fmaf_rn(b.x, w.x, -__fmul_rn(b.y, w.y)), __fmaf_rn(b.x, w.y, __fmul_rn(b.y, w.x)));
}
// acc + a * b
template <typename C>
__device__ __forceinline__ C cfma(C a, C b, C acc) {
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
    return acc;
}
__device__ __forceinline__ double2 mul_conj(double2 a, double2 b) {  // a * conj(b)
    return make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ void sincospi_r(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ void sincospi_r(double x, double* s, double* c) { sincospi(x, s, c); }

// Sample loads are cached in L2 only: the sigma-strided gather touches one 32-byte sector per sample
// and an L1 fill would fetch the whole 128-byte line.
// Request s of a launch: its signal row, its seed and the request index its random draws use.
// xmask: a permuted sample index p (already reduced mod n, or a uint32 product, n | 2^32) reads
// x[p & xmask]: n - 1, or period - 1 for a periodic extension.
struct ReqView {
    const void* x;
    uint64_t seed;
    uint32_t id;
    uint32_t xmask;
};
__device__ __forceinline__ ReqView req_view(const ReqDesc* reqs, const void* x, uint64_t row_bytes, uint64_t seed,
                                            uint32_t s, uint32_t nmask) {
    if (reqs) {
        const ReqDesc d = reqs[s];
        return ReqView{d.x, d.seed, d.id, d.period ? d.period - 1u : nmask};
    }
    return ReqView{static_cast<const unsigned char*>(x) + (size_t)s * row_bytes, seed, s, nmask};
}

__device__ __forceinline__ float2 ldg_c(const float2* p) { return __ldcg(p); }
__device__ __forceinline__ double2 ldg_c(const double2* p) { return __ldcg(p); }

// Precision of the decode.  Bins, subtraction sums, values and all index arithmetic are FP64.  The
// transcendental functions (the subtraction twiddles w^{a sigma i}, phases and magnitudes) run in
// the precision R of the data path: an FP32 bin carries ~1e-6 of accumulated rounding, so an FP32
// atan2 or sincospi (~1e-7) adds nothing measurable, while GB300's FP64 pipe is ~1/64 of FP32.
// Every phase the decode compares keeps a tolerance of at least tau_dec (1e-4 rad by default).

// w^e = exp(-2 pi i e / n) for an exact exponent e in [0, n), evaluated in precision R
template <typename R>
__device__ __forceinline__ double2 root_pow(uint32_t e, uint32_t nmask) {
    const uint32_t n = nmask + 1u;
    const int64_t es = e > (nmask >> 1) ? (int64_t)e - (int64_t)n : (int64_t)e;
    R s, c;
    sincospi_r((R)(2 * es) / (R)n, &s, &c);
    return make_double2((double)c, -(double)s);
}

// w^e = exp(-2 pi i e / n) for an exact exponent e in [0, n) from two tables of FP64 factors,
// exp(-2 pi i (e mod 2^sh) / n) and exp(-2 pi i 2^sh (e >> sh) / n): one complex product (a few ulp
// from a direct evaluation) instead of an FP64 sincospi, which GB300 runs at 1/64 of the FP32 rate
__device__ __forceinline__ double2 root_pow_tab(uint32_t e, const double2* tw, uint32_t sh) {
    const double2 lo = tw[e & ((1u << sh) - 1u)], hi = tw[(1u << sh) + (e >> sh)];
    return make_double2(hi.x * lo.x - hi.y * lo.y, hi.x * lo.y + hi.y * lo.x);
}

// The same from tables whose first part holds the factors minus one: w^e = h + h (l - 1), where the small
// second term's rounding is lost in the sum's (error below 1 ulp, against 2 of the plain product).
__device__ __forceinline__ double2 root_pow_fine(uint32_t e, const double2* tw, uint32_t sh) {
    const double2 d = tw[e & ((1u << sh) - 1u)], h = tw[(1u << sh) + (e >> sh)];
    return make_double2(fma(h.x, d.x, fma(-h.y, d.y, h.x)), fma(h.x, d.y, fma(h.y, d.x, h.y)));
}

// phase(z) / 2 pi in [0, 1)
__device__ __forceinline__ double phase01(double2 z) {
    double p = __ddiv_rn(atan2(z.y, z.x), 6.283185307179586476925286766559);
    if (p < 0.0) p += 1.0;
    if (p >= 1.0) p -= 1.0;
    return p;
}

// a * conj(b) with every product and sum rounded separately (no fused multiply-add), so that a
// decision taken on the result sees the same double an unfused host computation produces
__device__ __forceinline__ double2 mul_conj_rn(double2 a, double2 b) {
    return make_double2(__dadd_rn(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)),
                        __dsub_rn(__dmul_rn(a.y, b.x), __dmul_rn(a.x, b.y)));
}
__device__ __forceinline__ double cmag(double2 z) { return hypot(z.x, z.y); }
__device__ __forceinline__ uint32_t ilog2_u32(uint32_t v) { return 31u - __clz(v); }

// ------------------------------------------------------------------------------------------------
// block-wide helpers (kThreads threads)
// ------------------------------------------------------------------------------------------------
// Exclusive prefix sum of v[0..len) in place; returns the total.  tmp holds kThreads + 1 words.
__device__ inline uint32_t block_exclusive_scan(uint32_t* v, uint32_t len, uint32_t* tmp) {
    const uint32_t tid = threadIdx.x;
    const uint32_t seg = (len + kThreads - 1) / kThreads;
    const uint32_t b0 = min(len, tid * seg), b1 = min(len, b0 + seg);
    uint32_t sum = 0;
    for (uint32_t i = b0; i < b1; ++i) sum += v[i];
    // inclusive scan of the per-thread sums: within each warp by shuffles, then across the 8 warps
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (uint32_t off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) tmp[warp] = incl;
    __syncthreads();
    if (tid == 0) {
        uint32_t run = 0;
        for (uint32_t w = 0; w < (uint32_t)kThreads / 32u; ++w) {
            const uint32_t x = tmp[w];
            tmp[w] = run;
            run += x;
        }
        tmp[kThreads] = run;
    }
    __syncthreads();
    uint32_t run = tmp[warp] + incl - sum;
    for (uint32_t i = b0; i < b1; ++i) {
        const uint32_t x = v[i];
        v[i] = run;
        run += x;
    }
    const uint32_t total = tmp[kThreads];
    __syncthreads();
    return total;
}

// number of entries of the ascending array a[0..len) that are < key (lower) or <= key (upper)
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t* a, uint32_t len, uint32_t key) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ uint32_t upper_bound_u32(const uint32_t* a, uint32_t len, uint32_t key) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] <= key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Candidates (distinct indices, any order) sorted by index into (srt_idx, srt_val) by rank counting.
__device__ inline void rank_sort(const uint32_t* idx, const double2* val, uint32_t m, uint32_t* srt_idx, double2* srt_val) {
    for (uint32_t c = threadIdx.x; c < m; c += kThreads) {
        const uint32_t key = idx[c];
        uint32_t r = 0;
        for (uint32_t q = 0; q < m; ++q) r += idx[q] < key ? 1u : 0u;
        srt_idx[r] = key;
        srt_val[r] = val[c];
    }
    __syncthreads();
}

// In-place radix-2 decimation-in-time FFTs of H rows of B = 2^logB points held in bit-reversed
// order: a_j <- sum_r a_r exp(-2 pi i j r / B) in natural order (Lemma "hashtobins", step 3).
// The first min(5, logB) stages pair elements less than 32 apart: each warp holds 32 consecutive
// elements (one per lane) and exchanges partners by shuffles, with the twiddles exp(-i pi k / 16),
// k < 16, computed once per lane and shuffled to where they are needed.  The remaining stages run
// in place in shared memory, all rows together, one barrier per stage.  Butterfly arithmetic and
// twiddle values are the same in both forms.  Ends with a barrier.
template <typename R>
__device__ __forceinline__ void fft_first_stages(typename Cx<R>::T* a, uint32_t H, uint32_t logB) {
    using C = typename Cx<R>::T;
    const uint32_t B = 1u << logB;
    const uint32_t total = H * B, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t S = logB < 5 ? logB : 5;
    __syncthreads();  // the rows are in place
    {
        R ts, tc;
        sincospi_r(-(R)(lane & 15u) / (R)16, &ts, &tc);  // exp(-i pi k / 16), k = lane mod 16
        for (uint32_t g0 = warp * 32u; g0 < total; g0 += (uint32_t)kThreads) {
            const uint32_t i = g0 + lane;
            C v = i < total ? a[i] : mkc((R)0, (R)0);
            for (uint32_t st = 1; st <= S; ++st) {
                const uint32_t half = 1u << (st - 1);
                const uint32_t pos = lane & (half - 1);
                C w;
                w.x = __shfl_sync(0xffffffffu, tc, (int)(pos << (5 - st)));
                w.y = __shfl_sync(0xffffffffu, ts, (int)(pos << (5 - st)));
                C p;
                p.x = __shfl_xor_sync(0xffffffffu, v.x, (int)half);
                p.y = __shfl_xor_sync(0xffffffffu, v.y, (int)half);
                const bool upper = (lane & half) != 0;
                const C bv = cmul(upper ? v : p, w);
                const C av = upper ? p : v;
                v = upper ? csub(av, bv) : cadd(av, bv);
            }
            if (i < total) a[i] = v;
        }
    }
    __syncthreads();
}

template <typename R>
__device__ void block_fft_rows(typename Cx<R>::T* a, uint32_t H, uint32_t logB) {
    using C = typename Cx<R>::T;
    const uint32_t B = 1u << logB;
    const uint32_t halfB = B >> 1;
    fft_first_stages<R>(a, H, logB);
    const uint32_t S = logB < 5 ? logB : 5;
    for (uint32_t st = S + 1; st <= logB; ++st) {
        const uint32_t half = 1u << (st - 1);
        for (uint32_t idx = threadIdx.x; idx < H * halfB; idx += kThreads) {
            const uint32_t h = idx >> (logB - 1);
            const uint32_t k = idx & (halfB - 1);
            const uint32_t pos = k & (half - 1);
            const uint32_t i0 = h * B + ((k >> (st - 1)) << st) + pos;
            const uint32_t i1 = i0 + half;
            R sn, cs;
            sincospi_r(-(R)pos / (R)half, &sn, &cs);
            const C w = mkc(cs, sn);
            const C bv = cmul(a[i1], w);
            const C av = a[i0];
            a[i0] = cadd(av, bv);
            a[i1] = csub(av, bv);
        }
        __syncthreads();
    }
}

// block_fft_rows in FP64 with its twiddles from the factor tables (n = 2^logn): an FP64 sincospi costs
// about 45 operations of a pipe that issues at 1/64 of the FP32 rate, a butterfly 8, and thread pairs
// that exchange by shuffles would each form the whole product.  exp(-i pi pos / half) = w^{pos n / (2 half)}.
__device__ inline void fft_rows_fp64(double2* a, uint32_t H, uint32_t logB, uint32_t logn, const double2* tw, uint32_t sh) {
    const uint32_t halfB = (1u << logB) >> 1;
    __syncthreads();
    for (uint32_t st = 1; st <= logB; ++st) {
        const uint32_t half = 1u << (st - 1);
        for (uint32_t idx = threadIdx.x; idx < H * halfB; idx += kThreads) {
            const uint32_t h = idx >> (logB - 1), k = idx & (halfB - 1), pos = k & (half - 1);
            const uint32_t i0 = (h << logB) + ((k >> (st - 1)) << st) + pos, i1 = i0 + half, e = pos << (logn - st);
            const double2 w = logn - st >= sh ? tw[(1u << sh) + (e >> sh)] : root_pow_fine(e, tw, sh);
            const double2 b = a[i1], av = a[i0];
            const double2 bv = make_double2(b.x * w.x - b.y * w.y, b.x * w.y + b.y * w.x);
            a[i0] = cadd(av, bv);
            a[i1] = csub(av, bv);
        }
        __syncthreads();
    }
}

// dst[0..len) <- src[0..len) (another CTA's stores), eight loads in flight per thread
template <typename C>
__device__ __forceinline__ void load_rows(C* dst, const C* src, uint32_t len) {
    constexpr uint32_t N = sizeof(C) == 8 ? 8 : 4;
    for (uint32_t i0 = threadIdx.x; i0 < len; i0 += kThreads * N) {
        C v[N];
#pragma unroll
        for (uint32_t q = 0; q < N; ++q)
            if (i0 + q * kThreads < len) v[q] = __ldcg(src + i0 + q * kThreads);
#pragma unroll
        for (uint32_t q = 0; q < N; ++q)
            if (i0 + q * kThreads < len) dst[i0 + q * kThreads] = v[q];
    }
}

// Stages st + 1 .. st + N of an FFT of H rows: a thread takes the 2^N elements those stages mix, so that
// one pass over shared memory and one barrier serve N stages.  Ends with a barrier.
template <int N>
__device__ __forceinline__ void fft_pass(float2* a, uint32_t H, uint32_t logB, uint32_t st) {
    constexpr int M = 1 << N;
    const uint32_t half = 1u << st, groups = 1u << (logB - N);
    auto butterflies = [&](float2* row, const float2* w) {
        float2 v[M];
#pragma unroll
        for (int e = 0; e < M; ++e) v[e] = row[(uint32_t)e << st];
#pragma unroll
        for (int k = 0; k < N; ++k)
#pragma unroll
            for (int e = 0; e < M; ++e)
                if (!(e & (1 << k))) {
                    const float2 bv = cmul_rn(v[e | (1 << k)], w[(1 << k) - 1 + (e & ((1 << k) - 1))]);
                    const float2 av = v[e];
                    v[e] = cadd(av, bv);
                    v[e | (1 << k)] = csub(av, bv);
                }
#pragma unroll
        for (int e = 0; e < M; ++e) row[(uint32_t)e << st] = v[e];
    };
    // the twiddles of stage st + 1 + k at position lo: exp(-i pi (lo + f half) / (half 2^k)), f < 2^k
    auto twiddles = [&](uint32_t lo, float2* w) {
#pragma unroll
        for (int k = 0; k < N; ++k)
#pragma unroll
            for (int f = 0; f < (1 << k); ++f) {
                float sn, cs;  // (a quotient by a power of two: the product with its inverse is exact)
                sincospif(-(float)(lo + ((uint32_t)f << st)) * __int_as_float((int)(127u - st - (uint32_t)k) << 23), &sn, &cs);
                w[(1 << k) - 1 + f] = mkc(cs, sn);
            }
    };
    float2 w[M - 1];
    if (groups >= (uint32_t)kThreads) {  // every thread has a position: its twiddles serve all rows
        for (uint32_t q = threadIdx.x; q < groups; q += kThreads) {
            const uint32_t lo = q & (half - 1);
            twiddles(lo, w);
            for (uint32_t h = 0; h < H; ++h) butterflies(a + (h << logB) + ((q >> st) << (st + N)) + lo, w);
        }
    } else {
        for (uint32_t i = threadIdx.x; i < H * groups; i += kThreads) {
            const uint32_t h = i >> (logB - N), q = i & (groups - 1), lo = q & (half - 1);
            twiddles(lo, w);
            butterflies(a + (h << logB) + ((q >> st) << (st + N)) + lo, w);
        }
    }
    __syncthreads();
}

// The first five stages of rows of 32 or more elements (fft_first_stages, four groups of 32 elements per
// warp at a time: the shuffles of one group hide those of the others).
__device__ __forceinline__ void fft_first_five(float2* a, uint32_t total) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    __syncthreads();  // the rows are in place
    float ts, tc;
    sincospif(-(float)(lane & 15u) / 16.0f, &ts, &tc);  // exp(-i pi k / 16), k = lane mod 16
    float2 w[5];
#pragma unroll
    for (int st = 1; st <= 5; ++st) {
        const int pos = (int)(lane & ((1u << (st - 1)) - 1u));
        w[st - 1] = make_float2(__shfl_sync(0xffffffffu, tc, pos << (5 - st)), __shfl_sync(0xffffffffu, ts, pos << (5 - st)));
    }
    constexpr uint32_t G = 4;
    for (uint32_t g0 = warp * 32u; g0 < total; g0 += (uint32_t)kThreads * G) {
        float2 v[G];
#pragma unroll
        for (uint32_t g = 0; g < G; ++g)
            v[g] = g0 + g * kThreads < total ? a[g0 + g * kThreads + lane] : make_float2(0.f, 0.f);
#pragma unroll
        for (int st = 1; st <= 5; ++st) {
            const int half = 1 << (st - 1);
            const bool upper = (lane & (uint32_t)half) != 0;
#pragma unroll
            for (uint32_t g = 0; g < G; ++g) {
                const float2 p = make_float2(__shfl_xor_sync(0xffffffffu, v[g].x, half), __shfl_xor_sync(0xffffffffu, v[g].y, half));
                const float2 bv = cmul_rn(upper ? v[g] : p, w[st - 1]), av = upper ? p : v[g];
                v[g] = upper ? make_float2(__fsub_rn(av.x, bv.x), __fsub_rn(av.y, bv.y))
                             : make_float2(__fadd_rn(av.x, bv.x), __fadd_rn(av.y, bv.y));
            }
        }
#pragma unroll
        for (uint32_t g = 0; g < G; ++g)
            if (g0 + g * kThreads < total) a[g0 + g * kThreads + lane] = v[g];
    }
    __syncthreads();
}

// block_fft_rows with the stages past the fifth taken two or three per pass: as many as leave every
// thread a group of elements (B = 2048, two rows: two barriers instead of six, and a third of the
// sincospif).  The same butterflies, so the same bits.
__device__ inline void fft_rows_by_passes(float2* a, uint32_t H, uint32_t logB) {
    if (logB >= 5)
        fft_first_five(a, H << logB);
    else
        fft_first_stages<float>(a, H, logB);
    for (uint32_t st = logB < 5 ? logB : 5; st < logB;) {
        const uint32_t left = logB - st;
        if (left >= 3 && left != 4 && (H << (logB - 3)) >= (uint32_t)kThreads) {
            fft_pass<3>(a, H, logB, st);
            st += 3;
        } else if (left >= 2 && (H << (logB - 2)) >= (uint32_t)kThreads) {
            fft_pass<2>(a, H, logB, st);
            st += 2;
        } else {
            fft_pass<1>(a, H, logB, st);
            st += 1;
        }
    }
}

// the next array of a shared-memory layout: its offset (16-byte aligned)
__host__ __device__ inline size_t smem_take(size_t* off, size_t bytes) {
    const size_t o = (*off + 15) & ~size_t(15);
    *off = o + bytes;
    return o;
}
// warps that count (each with its own counters): 8 up to B = 1024
__host__ __device__ inline uint32_t split_segments(uint32_t B) { return B <= 1024 ? 8u : 8192u / B; }
// Stable counting split, in a CTA: per-warp counters, no sort.  place[e] <- the rank of entry e in (bin, index) order, from place[e] = its bin; start[j] <- the first
// rank of bin j (start[B] = nz).  cnt: split_segments(B) x B counters.
__device__ __forceinline__ void split_by_bin(uint32_t* place, uint32_t nz, uint32_t B, uint16_t* cnt, uint32_t* start, uint32_t* scan) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nseg = split_segments(B);
    for (uint32_t i = tid; i < nseg * B / 2; i += kThreads) reinterpret_cast<uint32_t*>(cnt)[i] = 0;
    __syncthreads();
    const uint32_t per = ((nz + nseg - 1) / nseg + 31u) & ~31u, beg = warp * per, end = min(nz, beg + per);
    uint16_t* mine = cnt + (size_t)warp * B;
    if (warp < nseg)
        for (uint32_t e0 = beg; e0 < end; e0 += 32) {
            const bool in = e0 + lane < end;
            const uint32_t b = in ? place[e0 + lane] : kNoIndex;
            const unsigned same = __match_any_sync(0xffffffffu, b);
            if (in && lane == (uint32_t)__ffs((int)same) - 1u) mine[b] = (uint16_t)(mine[b] + __popc((int)same));
            __syncwarp();
        }
    __syncthreads();
    for (uint32_t j = tid; j < B; j += kThreads) {
        uint32_t run = 0;
        for (uint32_t w = 0; w < nseg; ++w) {
            const uint32_t c = cnt[w * B + j];
            cnt[w * B + j] = (uint16_t)run;
            run += c;
        }
        start[j] = run;
    }
    __syncthreads();
    block_exclusive_scan(start, B, scan);  // ends with a barrier
    if (tid == 0) start[B] = nz;
    if (warp < nseg)
        for (uint32_t e0 = beg; e0 < end; e0 += 32) {
            const bool in = e0 + lane < end;
            const uint32_t b = in ? place[e0 + lane] : kNoIndex;
            const unsigned same = __match_any_sync(0xffffffffu, b);
            uint32_t base = 0;
            if (in) {
                base = mine[b];
                place[e0 + lane] = start[b] + base + (uint32_t)__popc((int)(same & ((1u << lane) - 1u)));
            }
            __syncwarp();
            if (in && lane == (uint32_t)__ffs((int)same) - 1u) mine[b] = (uint16_t)(base + __popc((int)same));
            __syncwarp();
        }
    __syncthreads();
}

// Bucket the nz entries of zhat by bin: bin_start[B+1] (exclusive prefix), bin_list (entry ids of
// each bin, ascending).  ent_bin must be filled.
__device__ inline void bucket_entries(const uint32_t* ent_bin, uint32_t nz, uint32_t B, uint32_t* bin_cnt,
                               uint32_t* bin_start, uint32_t* bin_list, uint32_t* scan_tmp) {
    if (nz == 0) {  // no entries: every bin list is empty
        for (uint32_t j = threadIdx.x; j <= B; j += kThreads) bin_start[j] = 0;
        __syncthreads();
        return;
    }
    if (nz <= (uint32_t)kThreads) {
        // one entry per thread: its place in bin_list is the number of entries before it in (bin, id)
        // order; scan_tmp receives the bins in that order, and bin_start[j] counts those below j
        if (threadIdx.x < nz) {
            const uint32_t e0 = threadIdx.x, b0 = ent_bin[e0];
            uint32_t r = 0;
            for (uint32_t e = 0; e < nz; ++e) {
                const uint32_t be = ent_bin[e];
                r += (be < b0 || (be == b0 && e < e0)) ? 1u : 0u;
            }
            bin_list[r] = e0;
            scan_tmp[r] = b0;
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j <= B; j += kThreads) bin_start[j] = lower_bound_u32(scan_tmp, nz, j);
        __syncthreads();
        return;
    }
    for (uint32_t j = threadIdx.x; j <= B; j += kThreads) bin_cnt[j] = 0;
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < nz; e += kThreads) atomicAdd(&bin_cnt[ent_bin[e]], 1u);
    __syncthreads();
    for (uint32_t j = threadIdx.x; j <= B; j += kThreads) bin_start[j] = bin_cnt[j];
    __syncthreads();
    block_exclusive_scan(bin_start, B + 1, scan_tmp);
    for (uint32_t j = threadIdx.x; j <= B; j += kThreads) bin_cnt[j] = bin_start[j];  // fill cursor
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < nz; e += kThreads) {
        const uint32_t slot = atomicAdd(&bin_cnt[ent_bin[e]], 1u);
        bin_list[slot] = e;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < B; j += kThreads) {  // insertion sort of each (short) bin list
        const uint32_t b0 = bin_start[j], b1 = bin_start[j + 1];
        for (uint32_t x = b0 + 1; x < b1; ++x) {
            const uint32_t v = bin_list[x];
            uint32_t y = x;
            while (y > b0 && bin_list[y - 1] > v) {
                bin_list[y] = bin_list[y - 1];
                --y;
            }
            bin_list[y] = v;
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------------------
// CTA arrival
// ------------------------------------------------------------------------------------------------
// Arrival of this CTA at a counter whose last arrival (the target-th) does the follow-up work.
// Returns 1 in every thread of the last arriving CTA.  Only thread 0 fences: the barrier before its
// fence orders every thread's stores before it (the fence is cumulative), and the barrier after it
// orders its fence before every thread's loads (the same pattern as a grid-wide barrier).  Data
// written by other CTAs of the same launch is then read through L2 (ld.global.cg).
// ---- bulk asynchronous copies (TMA, cp.async.bulk) completing on a shared-memory mbarrier ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");  // visible to the async proxy
}
// one arrival that also announces `bytes` of copies to complete in the current phase
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// global -> shared copy of `bytes` (a multiple of 16; both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Bounded wait for the phase of parity `parity`: true once it has completed, false after `limit`
// tries (each try may suspend the thread for a short, hardware-defined time).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
    for (uint32_t i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if (i > 64) __nanosleep(64);
    }
    return false;
}

__device__ __forceinline__ uint32_t arrive(uint32_t* counter, uint32_t target) {
    __shared__ uint32_t s_arrive_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t last = atomicAdd(counter, 1u) + 1u == target ? 1u : 0u;
        if (last) __threadfence();
        s_arrive_last = last;
    }
    __syncthreads();
    return s_arrive_last;
}

// an acquire load of *p (gpu scope) compared with v
__device__ __forceinline__ bool acquire_is(const uint32_t* p, uint32_t v) {
    uint32_t seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(p) : "memory");
    return seen == v;
}

// Arrival of one of two parties.  When an acquire load already sees the other party's arrival, this
// CTA is the last: the other party's writes are visible through the load, and nobody reads this CTA's
// writes through the counter, so the release fence and the atomic are skipped (the counter stays at 1
// until the caller clears it).  Otherwise as arrive(counter, 2).
__device__ __forceinline__ uint32_t arrive_pair(uint32_t* counter) {
    __shared__ uint32_t s_pair_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
        uint32_t last = 1u;
        if (seen != 1u) {
            __threadfence();
            last = atomicAdd(counter, 1u) + 1u == 2u ? 1u : 0u;
            if (last) __threadfence();
        }
        s_pair_last = last;
    }
    __syncthreads();
    return s_pair_last;
}

}  // namespace sfft
