// sfft_general.cu -- the general-case sparse FFT on sm_103a (Algorithms 2 and 3 of Hassanieh, Indyk,
// Katabi, Price): SparseFFT's rounds of LocateSignal (LocateInner votes over D_max levels) and
// EstimateValues (medians over R_est hashings, top-k'), for a batch of requests.
//
// The hashings of one round are non-adaptive (the intuition of Sec. 4.1): every LocateInner pair
// (a, a + beta) of every level and every EstimateValues hashing is known before any vote is counted.
// Nor do the samples of any round depend on zhat.  So a batch is one gather for all rounds, then three
// launches per round:
//   0. k_gen_permute  (rounds whose LocateInner pairs gather >= 2n samples) every request: x_{sigma m}
//                     for all m under the round's sigma, so that the pairs read it in order;
//   1. k_gen_gather   every (round, residue block, hashings, request): permuted gather, window,
//                     modulation, fold mod B (HashToBins steps 1-2);
//   2. k_gen_finish   every (hashing group, request): the fold's B-point FFT
//                     (step 3), recovered coefficients subtracted in FP64 (step 4), bins stored;
//                     for a LocateInner pair also c_j = phase(u_j / u'_j);
//   3. k_gen_locate   every (bin, request), t threads per bin (one per subregion): LocateSignal's
//                     levels in order, votes, regions, the bin's candidate for the list L and
//                     EstimateValues' medians of it;
//   4. k_gen_select   every request: the distinct candidates' top k', zhat += w_J.
// Reductions run in a fixed order; results are bit-reproducible.
#include <cuda_runtime.h>

#include <mutex>
#include <stdint.h>

#include "philox.cuh"
#include "sfft_device.cuh"
#include "sfft_internal.h"

namespace sfft {

// ------------------------------------------------------------------------------------------------
// hashing parameters
// ------------------------------------------------------------------------------------------------
struct HashDesc {
    uint32_t sigma, b, H;
    uint32_t a[2];
    uint64_t beta;
};

// LocateSignal's sigma, b of round r (Algorithm 3: one draw per call)
__device__ __forceinline__ void locate_sigma_b(uint64_t seed, uint32_t s, uint32_t r, uint32_t nmask, uint32_t* sigma,
                                               uint32_t* b) {
    const Words4 w = draw(seed, s, r, 0, kKindLocate);
    *sigma = (w.w[0] & nmask) | 1u;
    *b = w.w[1] & nmask;
}

// LocateInner round q of level D (g = (D - 1) R_loc + q): a uniform on [n], beta uniform on the level's range
__device__ __forceinline__ void inner_a_beta(uint64_t seed, uint32_t s, uint32_t r, uint32_t g, uint32_t nmask,
                                             uint64_t lo, uint64_t hi, uint32_t* a, uint64_t* beta) {
    const Words4 w = draw(seed, s, r, g, kKindInner);
    *a = w.w[0] & nmask;
    *beta = lo + (((uint64_t)w.w[1] * (hi - lo + 1)) >> 32);
}

// Group g of a round: g < npairs is LocateInner pair g (hashings a and a + beta under the round's
// sigma, b); g >= npairs is EstimateValues hashing q = g - npairs with fresh (sigma_q, a_q, b_q).
__device__ __forceinline__ HashDesc group_desc(const GenArgs& a, uint64_t seed, uint32_t id, uint32_t g) {
    HashDesc h;
    if (g < a.npairs) {
        locate_sigma_b(seed, id, a.round, a.nmask, &h.sigma, &h.b);
        const uint32_t D = g / a.R_loc;
        inner_a_beta(seed, id, a.round, g, a.nmask, a.beta_lo[D], a.beta_hi[D], &h.a[0], &h.beta);
        h.a[1] = (uint32_t)((h.a[0] + h.beta) & a.nmask);
        h.H = 2;
    } else {
        const Words4 w = draw(seed, id, a.round, g - a.npairs, kKindEstimate);
        h.sigma = (w.w[0] & a.nmask) | 1u;
        h.b = w.w[1] & a.nmask;
        h.a[0] = w.w[2] & a.nmask;
        h.a[1] = 0;
        h.beta = 0;
        h.H = 1;
    }
    return h;
}

// request s of a general-mode launch (signal row, seed, draw index)
__device__ __forceinline__ ReqView gen_req(const GenArgs& a, uint32_t s) {
    return req_view(a.reqs, a.x, a.n * sizeof(float2), a.seed, s, a.nmask);
}

__device__ __forceinline__ uint32_t hash_index(const GenArgs& a, uint32_t g, uint32_t h) {
    return g < a.npairs ? 2 * g + h : 2 * a.npairs + (g - a.npairs);
}

// bin and offset of a permuted position (Sec. 3 definitions)
__device__ __forceinline__ int32_t gen_offset(uint32_t p, uint32_t n, uint32_t nmask, uint32_t logNp, uint32_t* jbin) {
    const uint32_t Np = 1u << logNp;
    const uint32_t jj = ((p + (Np >> 1)) & nmask) >> logNp;
    const uint32_t dd = (p - jj * Np) & nmask;
    *jbin = jj;
    return dd > (nmask >> 1) ? (int32_t)((int64_t)dd - (int64_t)n) : (int32_t)dd;
}

// Launches of one stream group follow one another with programmatic serialisation: a kernel may start when
// the CTAs of the one before have ended, without waiting for its memory to be flushed, and waits here before
// it reads or writes what that one did (each kernel waits, so it waits for all before).  One request at
// n = 2^18, k = 50: 109 us, was 131; n = 2^20, k = 500, batch 5: 562 us, was 602.
// a.early: a kernel also lets the next one start as soon as its own CTAs all run (see general_early).
__device__ __forceinline__ void after_previous(const GenArgs& a) {
    if (a.early) cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
}

// ------------------------------------------------------------------------------------------------
// 0. permuted copy (rounds whose LocateInner pairs gather >= 2n samples)
// ------------------------------------------------------------------------------------------------
// xperm[m] = x_{sigma m} for every m in [n], sigma the round's LocateInner sigma: the pairs then read
// x_{sigma (t - a)} = xperm[(t - a) mod n] in order.  Grid (CTAs, batch); 8 loads in flight per thread.
__global__ void __launch_bounds__(kThreads) k_gen_permute(const GenArgs a) {
    const uint32_t s = a.req_base + blockIdx.y;
    const ReqView rq = gen_req(a, s);
    uint32_t sigma, b;
    locate_sigma_b(rq.seed, rq.id, a.round, a.nmask, &sigma, &b);
    const float2* __restrict__ x = static_cast<const float2*>(rq.x);
    float2* __restrict__ xp = a.xperm + (size_t)s * a.n;
    constexpr uint32_t kPer = kThreads * 8;
    for (uint64_t m0 = (uint64_t)blockIdx.x * kPer; m0 < a.n; m0 += (uint64_t)gridDim.x * kPer) {
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint64_t m = m0 + (uint64_t)q * kThreads + threadIdx.x;
            if (m < a.n) v[q] = __ldcg(x + ((sigma * (uint32_t)m) & rq.xmask));
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint64_t m = m0 + (uint64_t)q * kThreads + threadIdx.x;
            if (m < a.n) xp[m] = v[q];
        }
    }
}

// ------------------------------------------------------------------------------------------------
// 1. gather and fold
// ------------------------------------------------------------------------------------------------
// A CTA owns kThreads residues mod B of NH hashings that share (sigma, b) -- the two of each of NH / 2
// LocateInner pairs, or one EstimateValues hashing -- and folds every tap of those residues, one
// residue per thread: no partial fold leaves the CTA.  Samples go from L2 or HBM straight to the
// thread that folds them (16 loads in flight each), and a tap's window product G_t w^{sigma b t} is
// formed once for the NH hashings.
// Measured against the form it replaces (four 2048-tap chunks per CTA staged in shared memory, partial
// folds of every CTA summed by the last to arrive), whole calls: n = 2^22, k = 256, batch 8: 1323 us,
// was 1552; n = 2^20, k = 500, batch 5: 1252 us, was 1797.  Bound by L2 (the pairs' in-order reads) or
// by random 32-byte sectors of HBM (long signals).
// Order of the sums: the window is cut into ranges of a.rtaps taps; a residue's taps of a range are
// accumulated in order from zero (B < kThreads: by the kThreads / B threads of the residue, whose sums
// are added in thread order), and the ranges' sums are added in range order.
template <int NH>
__device__ __forceinline__ void gather_residues(const GenArgs& a, const float2* __restrict__ x, uint32_t xmul,
                                                uint32_t xmask, uint32_t sb, const uint32_t* ah, uint32_t nh, uint32_t blk,
                                                float2* __restrict__ out, float2 (*red)[kThreads]) {
    constexpr int TB = NH >= 8 ? 2 : (NH == 4 ? 4 : (NH == 2 ? 8 : 16));  // taps per batch of loads
    const uint32_t tid = threadIdx.x, B = a.B;
    const uint32_t step = B > (uint32_t)kThreads ? B : (uint32_t)kThreads;  // a thread's taps are step apart
    const uint32_t first = blk * kThreads, k0 = first + tid;
    const uint32_t ntot = (uint32_t)(2 * a.T + 1);
    const uint32_t t0 = (uint32_t)(int32_t)(-a.T) + k0;  // first tap, mod 2^32
    const uint32_t nt = a.rtaps / step;                  // a thread's taps per range (a power of two if there are several)
    const bool several = ntot > a.rtaps;
    const uint32_t mend = first < ntot ? (ntot - first + step - 1) / step : 0;  // batches end here for every thread
    float2 acc[NH], sum[NH];
    uint32_t xi[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        acc[h] = sum[h] = make_float2(0.f, 0.f);
        xi[h] = xmul * (t0 - ah[h]);
    }
    const uint32_t xstep = xmul * step, estep = sb * step;
    uint32_t e0 = sb * t0;
    const float two_over_n = 2.0f / (float)a.n;
    auto end_range = [&]() {
        if (B >= (uint32_t)kThreads) {
#pragma unroll
            for (int h = 0; h < NH; ++h) sum[h] = cadd(sum[h], acc[h]);
        } else {
            // thread r < B owns residue (r - T) mod B: the threads r + i B folded its taps
#pragma unroll
            for (int h = 0; h < NH; ++h) red[h][tid] = acc[h];
            __syncthreads();
            if (tid < B)
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    float2 w = make_float2(0.f, 0.f);
                    for (uint32_t i = tid; i < (uint32_t)kThreads; i += B) w = cadd(w, red[h][i]);
                    sum[h] = cadd(sum[h], w);
                }
            __syncthreads();
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) acc[h] = make_float2(0.f, 0.f);
    };
    for (uint32_t m0 = 0; m0 < mend; m0 += TB) {
        float2 v[TB][NH];
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            const bool in = k0 + (m0 + (uint32_t)u) * step < ntot;
#pragma unroll
            for (int h = 0; h < NH; ++h)
                if (in) v[u][h] = __ldcg(x + ((xi[h] + (uint32_t)u * xstep) & xmask));
        }
        float2 gt[TB];
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            if (k0 + (m0 + (uint32_t)u) * step < ntot) {
                const int32_t t = (int32_t)(t0 + (m0 + (uint32_t)u) * step);
                const float gv = a.taps[t < 0 ? -t : t];
                const uint32_t e = (e0 + (uint32_t)u * estep) & a.nmask;
                const int32_t es = e > (a.nmask >> 1) ? (int32_t)((int64_t)e - (int64_t)a.n) : (int32_t)e;
                float sn, cs;
                sincospif((float)es * two_over_n, &sn, &cs);
                gt[u] = make_float2(gv * cs, -gv * sn);
            }
        }
#pragma unroll
        for (int u = 0; u < TB; ++u) {
            if (u % 2 == 0 && several && m0 + (uint32_t)u != 0 && ((m0 + (uint32_t)u) & (nt - 1)) == 0 &&
                m0 + (uint32_t)u < mend)  // nt >= 2
                end_range();
            if (k0 + (m0 + (uint32_t)u) * step < ntot) {
#pragma unroll
                for (int h = 0; h < NH; ++h) acc[h] = cfma(gt[u], v[u][h], acc[h]);
            }
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) xi[h] += (uint32_t)TB * xstep;
        e0 += (uint32_t)TB * estep;
    }
    end_range();
    if (B >= (uint32_t)kThreads || tid < B) {
        // in bit-reversed order, as the bin FFT takes them
        const uint32_t r = __brev(t0 & (B - 1)) >> (32u - a.logB);
#pragma unroll
        for (int h = 0; h < NH; ++h)
            if ((uint32_t)h < nh) out[(size_t)h * B + r] = sum[h];
    }
}

// P pairs from g0 on (the round's last block may hold fewer)
template <int P>
__device__ __forceinline__ void gather_pairs(const GenArgs& a, const ReqView& rq, uint32_t s, uint32_t g0, uint32_t blk,
                                             float2* part, float2 (*red)[kThreads]) {
    const uint32_t np = min((uint32_t)P, a.npairs - g0);
    // a round with a permuted copy reads xperm[(t - a) mod n] = x_{sigma (t - a)} in order
    const bool perm = a.xperm != nullptr;
    uint32_t sigma, b, ah[2 * P];
    locate_sigma_b(rq.seed, rq.id, a.round, a.nmask, &sigma, &b);
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const uint32_t g = g0 + min((uint32_t)p, np - 1), D = g / a.R_loc;  // past the last pair: it again, not stored
        uint64_t beta;
        inner_a_beta(rq.seed, rq.id, a.round, g, a.nmask, a.beta_lo[D], a.beta_hi[D], &ah[2 * p], &beta);
        ah[2 * p + 1] = (uint32_t)((ah[2 * p] + beta) & a.nmask);
    }
    gather_residues<2 * P>(a, perm ? a.xperm + (size_t)s * a.n : static_cast<const float2*>(rq.x), perm ? 1u : sigma,
                           perm ? a.nmask : rq.xmask, sigma * b, ah, 2 * np, blk, part + (size_t)g0 * 2 * a.B, red);
}

// Every round's hashings in one launch (their samples do not depend on zhat): grid (CTAs of all
// rounds, requests), request by request so that a signal and its copies stay in L2; a round's CTAs
// are its EstimateValues hashings, then its blocks of P pairs, residue blocks fastest.  The small
// rounds' few CTAs run beside the first round's.  Whole calls, against one gather per round (which plans near
// the memory limit still use): n = 2^22, k = 256, batch 8: 742 us, 922; n = 2^18, k = 50, one request: 109 us,
// 130; n = 2^20, k = 500, batch 5: 566 us, 601.  n = 2^26, k = 64, batch 4 reads 26.3 M random sectors of HBM
// at 44 G/s.
template <int NR>
struct GatherParams {
    uint32_t R;
    uint32_t seg[NR + 1];  // first CTA of each round
    uint32_t P[NR];        // pairs per CTA: 1, 2 or 4
    GenArgs r[NR];
};
template <int NR>
__global__ void __launch_bounds__(kThreads, 2) k_gen_gather(const __grid_constant__ GatherParams<NR> gp) {
    __shared__ float2 red[8][kThreads];
    uint32_t r = 0;
    while (r + 1 < gp.R && blockIdx.x >= gp.seg[r + 1]) ++r;
    const GenArgs& a = gp.r[r];
    const uint32_t s = a.req_base + blockIdx.y;
    const uint32_t blocks = a.B > (uint32_t)kThreads ? a.B / kThreads : 1u;
    const uint32_t local = blockIdx.x - gp.seg[r], blk = local % blocks, y = local / blocks;
    const ReqView rq = gen_req(a, s);
    float2* part = a.part + (size_t)s * a.part_stride;
    if (y < a.R_est) {
        const uint32_t g = a.npairs + y;
        const HashDesc h = group_desc(a, rq.seed, rq.id, g);
        after_previous(a);
        gather_residues<1>(a, static_cast<const float2*>(rq.x), h.sigma, rq.xmask, h.sigma * h.b, h.a, 1, blk,
                           part + (size_t)g * 2 * a.B, red);
        return;
    }
    const uint32_t P = gp.P[r], g0 = (y - a.R_est) * P;
    after_previous(a);  // the permuted copies
    if (P == 4)
        gather_pairs<4>(a, rq, s, g0, blk, part, red);
    else if (P == 2)
        gather_pairs<2>(a, rq, s, g0, blk, part, red);
    else
        gather_pairs<1>(a, rq, s, g0, blk, part, red);
}

// ------------------------------------------------------------------------------------------------
// 2. finish the bins of one hashing group
// ------------------------------------------------------------------------------------------------
// One CTA per (hashing group, request): the fold's B-point FFTs, then the recovered coefficients are
// subtracted in FP64, entry by entry in index order, and a pair's phases are formed.  zhat's entries
// are placed by bin with a stable counting split (per-warp counters, no sort), up to kFinSlab of them at
// a time, so that every array stays on chip whatever zhat holds.  Bound by latency in the first round,
// by FP64 (1/64 of the FP32 rate) once zhat has many entries: per entry and hashing four products, and
// one chain of subtractions per (bin, hashing, component).  Measured alone at n = 2^20, k = 500 (last
// round: 16 bins, about 2000 entries): 110 us before, with bin lists sorted by insertion, one thread
// per bin and arrays in device memory.  Whole calls: 943 -> 640 us there (batch 5), 1155 -> 963 us at
// n = 2^22, k = 256, batch 8.
constexpr uint32_t kFinSlab = 2048;  // entries of zhat handled at once (8 per thread)
constexpr uint32_t kFinPer = kFinSlab / kThreads;
struct GenFinLayout {
    size_t U, term, slot, cnt, start, ub, scan, total;
};
// nzmax: the most entries zhat can have when the round starts
__host__ __device__ inline GenFinLayout gen_fin_layout(uint32_t B, uint32_t nzmax) {
    GenFinLayout L;
    const uint32_t ns = nzmax < kFinSlab ? nzmax : kFinSlab;
    size_t off = 0;
    L.U = smem_take(&off, (size_t)2 * B * 8);
    L.term = smem_take(&off, (size_t)ns * 2 * 16);
    L.slot = smem_take(&off, (size_t)ns * 4);
    L.cnt = smem_take(&off, ns ? (size_t)split_segments(B) * B * 2 : 0);
    L.start = smem_take(&off, ns ? (size_t)(B + 1) * 4 : 0);
    L.ub = smem_take(&off, ns && B < (uint32_t)kThreads ? (size_t)4 * B * 8 : 0);
    L.scan = smem_take(&off, (size_t)(kThreads + 8) * 4);
    L.total = off;
    return L;
}
size_t general_finish_smem(uint32_t B, uint32_t nzmax) { return gen_fin_layout(B, nzmax).total; }

// (double)v, on the integer units for a zero or normal v
__device__ __forceinline__ double widen(float v) {
    const uint32_t f = __float_as_uint(v), m = f & 0x7FFFFFFFu;
    if (m - 0x00800000u >= 0x7F000000u && m != 0) return (double)v;  // denormal, infinite or NaN
    const uint32_t hi = (f & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(f << 29));
}
// a x + b y rounded once from a sum good to ~2^-46 (exact products, their sum and its error)
__device__ __forceinline__ float dot2(float a, float x, float b, float y) {
    const float p = __fmul_rn(a, x), pe = __fmaf_rn(a, x, -p);
    const float q = __fmul_rn(b, y), qe = __fmaf_rn(b, y, -q);
    const float s = __fadd_rn(p, q), t = __fsub_rn(s, p);
    const float e = __fadd_rn(__fsub_rn(p, __fsub_rn(s, t)), __fsub_rn(q, t));
    return __fadd_rn(s, __fadd_rn(e, __fadd_rn(pe, qe)));
}
// (z.x, z.y) for an FP32 arctangent: times a power of two where the larger part lies outside 2^-96 .. 2^124,
// where float loses it (signals scaled below about 1e-15 or above 1e18); the phase stays.
__device__ __forceinline__ float2 direction(double2 z) {
    const uint32_t hx = (uint32_t)__double2hiint(z.x) & 0x7FFFFFFFu, hy = (uint32_t)__double2hiint(z.y) & 0x7FFFFFFFu;
    const uint32_t e = max(hx, hy) >> 20;  // 1023 + the larger part's exponent
    if (e - 927u > 220u && e - 1u < 2045u) {
        const double scale = __hiloint2double((int)((2046u - e) << 20), 0);
        z.x *= scale;
        z.y *= scale;
    }
    return make_float2((float)z.x, (float)z.y);
}

__global__ void __launch_bounds__(kThreads) k_gen_finish(const GenArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t s = a.req_base + blockIdx.y, g = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ReqView rq = gen_req(a, s);
    const HashDesc h = group_desc(a, rq.seed, rq.id, g);
    const uint32_t B = a.B;
    const GenFinLayout Ly = gen_fin_layout(B, a.nzmax);
    float2* U = reinterpret_cast<float2*>(smem + Ly.U);
    double2* term = reinterpret_cast<double2*>(smem + Ly.term);       // [slot][2]: by bin, then by index
    uint32_t* slot = reinterpret_cast<uint32_t*>(smem + Ly.slot);     // an entry's bin, then its place in term
    uint16_t* cnt = reinterpret_cast<uint16_t*>(smem + Ly.cnt);       // [segment][B]
    uint32_t* start = reinterpret_cast<uint32_t*>(smem + Ly.start);   // first place of each bin
    double* ub = reinterpret_cast<double*>(smem + Ly.ub);             // B < kThreads: [hashing][component][B]
    uint32_t* scan = reinterpret_cast<uint32_t*>(smem + Ly.scan);
    const uint32_t logNp = (uint32_t)(63 - __clzll((long long)a.n)) - a.logB;
    after_previous(a);
    // step 3: the fold (bit-reversed), B-point FFT per hashing
    load_rows(U, a.part + (size_t)s * a.part_stride + (size_t)g * 2 * B, h.H * B);
    const uint32_t nz = min(a.zcount[s], a.nzmax);
    const uint32_t* zidx = a.zidx + (size_t)s * a.zcap;
    const double2* zval = a.zval + (size_t)s * a.zcap;
    fft_rows_by_passes(U, h.H, a.logB);
    double2* bins = a.bins + (size_t)s * a.bins_stride;
    uint32_t* phase = a.phase + (size_t)s * a.phase_stride + (size_t)g * B;
    const float two_over_n = 2.0f / (float)a.n;
    const uint32_t row0 = hash_index(a, g, 0);
    // a bin after the last entry: stored, and c_j for a pair: an FP32 arctangent of the product
    // u_j conj(u'_j) (the vote arcs are s pi wide and the FP32 bins carry ~1e-6 of phase noise), in units
    // of 2^-32 of a turn; z is the product rounded to float
    auto store_phase = [&](uint32_t j, float2 z) {
        phase[j] = (uint32_t)__double2int_rn(widen(atan2f(z.y, z.x)) * (4294967296.0 * 0.15915494309189533576888));
    };
    if (nz == 0) {
        for (uint32_t j = tid; j < B; j += kThreads) {
            const float2 u = U[j];
            bins[(size_t)row0 * B + j] = make_double2(widen(u.x), widen(u.y));
            if (h.H == 2) {
                const float2 v = U[B + j];
                bins[(size_t)(row0 + 1) * B + j] = make_double2(widen(v.x), widen(v.y));
                float2 z = make_float2(dot2(u.x, v.x, u.y, v.y), dot2(u.y, v.x, -u.x, v.y));
                const float mag = fabsf(z.x) + fabsf(z.y);
                if (!(mag > 1e-30f && mag < 1e38f))  // beyond the range of the exact products' errors
                    z = direction(mul_conj_rn(make_double2(widen(u.x), widen(u.y)), make_double2(widen(v.x), widen(v.y))));
                store_phase(j, z);
            }
        }
        return;
    }
    const uint32_t slab = min(a.nzmax, kFinSlab);
    for (uint32_t z0 = 0; z0 < nz; z0 += slab) {
        const uint32_t m = min(slab, nz - z0);
        const bool first = z0 == 0, last = z0 + m == nz;
        // step 4 terms: W(-o(i)) zhat_i w^{a_h sigma i}
        double2 gz[kFinPer];
        uint32_t si[kFinPer];
#pragma unroll
        for (uint32_t q = 0; q < kFinPer; ++q) {
            const uint32_t e = tid + q * kThreads;
            if (e < m) {
                const uint32_t i = zidx[z0 + e];
                uint32_t jb;
                const int32_t o = gen_offset((h.sigma * (i - h.b)) & a.nmask, (uint32_t)a.n, a.nmask, logNp, &jb);
                slot[e] = jb;
                si[q] = h.sigma * i;
                const double gain = a.wtab[o < 0 ? -o : o];
                const double2 z = zval[z0 + e];
                gz[q] = make_double2(gain * z.x, gain * z.y);
            }
        }
        split_by_bin(slot, m, B, cnt, start, scan);  // (a barrier before it reads the slots)
#pragma unroll
        for (uint32_t q = 0; q < kFinPer; ++q) {
            const uint32_t e = tid + q * kThreads;
            if (e < m) {
                const uint32_t at = slot[e];
                for (uint32_t hh = 0; hh < h.H; ++hh) {
                    const uint32_t ex = (h.a[hh] * si[q]) & a.nmask;
                    const int32_t es = ex > (a.nmask >> 1) ? (int32_t)((int64_t)ex - (int64_t)a.n) : (int32_t)ex;
                    float sn, cs;
                    sincospif((float)es * two_over_n, &sn, &cs);
                    const double wx = widen(cs), wy = widen(-sn);
                    term[2 * at + hh] = make_double2(gz[q].x * wx - gz[q].y * wy, gz[q].x * wy + gz[q].y * wx);
                }
            }
        }
        __syncthreads();
        if (B < (uint32_t)kThreads) {
            // few bins with long lists: one thread per (component, hashing, bin)
            for (uint32_t i = tid; i < 2 * h.H * B; i += kThreads) {
                const uint32_t j = i & (B - 1), c = (i >> a.logB) & 1u, hh = i >> (a.logB + 1);
                const double* tc = reinterpret_cast<const double*>(term + hh) + c;
                double u = first ? widen(c ? U[hh * B + j].y : U[hh * B + j].x) : ub[i];
                for (uint32_t x = start[j], x1 = start[j + 1]; x < x1; ++x) u -= tc[4 * x];
                ub[i] = u;
            }
            __syncthreads();
            if (last)
                for (uint32_t j = tid; j < B; j += kThreads) {
                    const double2 u = make_double2(ub[j], ub[B + j]);
                    bins[(size_t)row0 * B + j] = u;
                    if (h.H == 2) {
                        const double2 v = make_double2(ub[2 * B + j], ub[3 * B + j]);
                        bins[(size_t)(row0 + 1) * B + j] = v;
                        store_phase(j, direction(mul_conj_rn(u, v)));
                    }
                }
        } else {
            for (uint32_t j = tid; j < B; j += kThreads) {
                const uint32_t x0 = start[j], x1 = start[j + 1];
                double2 u[2];
                for (uint32_t hh = 0; hh < h.H; ++hh) {
                    const float2 v = U[hh * B + j];
                    u[hh] = first ? make_double2(widen(v.x), widen(v.y)) : bins[(size_t)(row0 + hh) * B + j];
                }
                for (uint32_t x = x0; x < x1; ++x)
                    for (uint32_t hh = 0; hh < h.H; ++hh) {
                        const double2 t = term[2 * x + hh];
                        u[hh].x -= t.x;
                        u[hh].y -= t.y;
                    }
                for (uint32_t hh = 0; hh < h.H; ++hh) bins[(size_t)(row0 + hh) * B + j] = u[hh];
                if (h.H == 2 && last) {
                    store_phase(j, direction(mul_conj_rn(u[0], u[1])));
                }
            }
        }
        if (!last) __syncthreads();  // the arrays are filled again
    }
}

// ------------------------------------------------------------------------------------------------
// 3. LocateSignal: votes over the levels
// ------------------------------------------------------------------------------------------------
// One LocateInner vote test (Algorithm 3: |beta theta_{j,q} - c_j| circular < s pi).  f = e / M with
// e the exact fixed-point value of beta (m + sigma b) mod n and M = n 2^F.  The caller-bins entry takes
// the test on integers except for the (rare) e next to a boundary, where the double expression of the
// test decides, evaluated exactly as written.
struct VoteBounds {
    uint64_t ilo, len;    // e is inside iff (e - ilo) mod M <= len
    uint64_t amb0, amb1;  // integers within 0.25 of a boundary (or ~0 when none)
    double c;
};
constexpr int kVoteGuard = 16;  // extra fraction bits of the fixed-point boundaries
// Boundaries of the vote arc (c - s/2, c + s/2) in units of 1/M, as 64-bit fixed point with
// kVoteGuard fraction bits: c M 2^G is one exact scaling of c (truncated to an integer, an error
// below 2^-G units), so only one double operation is spent per (bin, round).
__device__ __forceinline__ VoteBounds vote_bounds(double c, int64_t hw_fix, uint32_t logM) {
    VoteBounds v;
    const int64_t one = int64_t(1) << kVoteGuard, frac_mask = one - 1;
    const int64_t xfix = (int64_t)(c * ldexp(1.0, (int)logM + kVoteGuard));
    const int64_t blf = xfix - hw_fix, bhf = xfix + hw_fix;
    const uint64_t mask = (uint64_t(1) << logM) - 1;
    const int64_t ilo = (blf >> kVoteGuard) + 1;                  // smallest integer > bl
    const int64_t ihi = ((bhf + frac_mask) >> kVoteGuard) - 1;    // largest integer < bh
    v.ilo = (uint64_t)ilo & mask;
    v.len = (uint64_t)(ihi - ilo) & mask;
    const int64_t fl = blf & frac_mask, fh = bhf & frac_mask;
    v.amb0 = fl < one / 4 ? ((uint64_t)(blf >> kVoteGuard) & mask)
                          : (fl > 3 * (one / 4) ? ((uint64_t)((blf >> kVoteGuard) + 1) & mask) : ~0ull);
    v.amb1 = fh < one / 4 ? ((uint64_t)(bhf >> kVoteGuard) & mask)
                          : (fh > 3 * (one / 4) ? ((uint64_t)((bhf >> kVoteGuard) + 1) & mask) : ~0ull);
    v.c = c;
    return v;
}
// The vote test on a given phase c, as written in Algorithm 3 (circular distance below s pi), in
// double precision.
__device__ __forceinline__ bool vote_hit_exact(double c, uint64_t e, uint64_t M, double s) {
    const double f = (double)e / (double)M;
    double dist = fabs(f - c);
    if (dist > 0.5) dist = 1.0 - dist;
    return dist < s / 2.0;
}
// half width s M / 2 of the vote arc in the same fixed point
__device__ __forceinline__ int64_t vote_halfwidth(double s, uint32_t logM) {
    return (int64_t)llrint(0.5 * s * ldexp(1.0, (int)logM + kVoteGuard));
}
__device__ __forceinline__ bool vote_hit(const VoteBounds& v, uint64_t e, uint64_t M, double s) {
    if (e == v.amb0 || e == v.amb1) return vote_hit_exact(v.c, e, M, s);
    return ((e - v.ilo) & (M - 1)) <= v.len;
}

// Votes of bin j at one level, then its region update (the four consecutive subregions with the
// most votes among those with a majority; bottom when no subregion has one).
// phase(q) returns c_j of LocateInner round q; beta[q] its beta.  T = t subregions, a compile-time
// constant so that the vote counters live in registers.
template <int T, typename PhaseFn>
__device__ __forceinline__ void locate_bin_t(uint32_t nrep, const uint64_t* beta, PhaseFn phase, uint64_t sb_fp,
                                             uint64_t w_fp, uint32_t logM, double s, int64_t hw_fix, uint64_t& l_fp,
                                             uint8_t& valid, uint32_t* votes_out) {
    uint32_t v[T];
#pragma unroll
    for (int q = 0; q < T; ++q) v[q] = 0;
    const uint64_t M = uint64_t(1) << logM;
    const uint64_t mask = M - 1;
    const uint64_t half_step = w_fp / (2 * (uint64_t)T), step = w_fp / T;
    for (uint32_t r = 0; r < nrep; ++r) {
        const VoteBounds vb = vote_bounds(phase(r), hw_fix, logM);
        // e_q = beta (m_q + sigma b) mod M, m_q = l + (2q - 1) w / 2t, advanced by beta w / t
        uint64_t e = (beta[r] * ((l_fp + half_step + sb_fp) & mask)) & mask;
        const uint64_t de = (beta[r] * step) & mask;
#pragma unroll
        for (int q = 0; q < T; ++q) {
            if (vote_hit(vb, e, M, s)) v[q] += 1;
            e = (e + de) & mask;
        }
    }
    if (votes_out) {
#pragma unroll
        for (int q = 0; q < T; ++q) votes_out[q] = v[q];
    }
    bool any = false;
#pragma unroll
    for (int q = 0; q < T; ++q) any = any || 2u * v[q] > nrep;
    if (!any) {
        valid = 0;
        return;
    }
    uint32_t best = 0, best_sum = 0;
#pragma unroll
    for (int q0 = 0; q0 + 4 <= T; ++q0) {
        const uint32_t sum = v[q0] + v[q0 + 1] + v[q0 + 2] + v[q0 + 3];
        if (q0 == 0 || sum > best_sum) {
            best = (uint32_t)q0;
            best_sum = sum;
        }
    }
    l_fp = (l_fp + (uint64_t)best * step) & mask;
}
template <typename PhaseFn>
__device__ void locate_bin(uint32_t t, uint32_t nrep, const uint64_t* beta, PhaseFn phase, uint64_t sb_fp,
                           uint64_t w_fp, uint32_t logM, double s, int64_t hw_fix, uint64_t& l_fp, uint8_t& valid,
                           uint32_t* votes_out) {
    // the schedule admits t in {8, 16, 32} (a power of two in [8, kMaxT])
    if (t == 8)
        locate_bin_t<8>(nrep, beta, phase, sb_fp, w_fp, logM, s, hw_fix, l_fp, valid, votes_out);
    else if (t == 16)
        locate_bin_t<16>(nrep, beta, phase, sb_fp, w_fp, logM, s, hw_fix, l_fp, valid, votes_out);
    else
        locate_bin_t<32>(nrep, beta, phase, sb_fp, w_fp, logM, s, hw_fix, l_fp, valid, votes_out);
}

// ------------------------------------------------------------------------------------------------
// EstimateValues on one candidate
// ------------------------------------------------------------------------------------------------
// w_i = median_q Re e_q + i median_q Im e_q over the hashings q whose window gain at i is >= est_gmin,
// e_q = u^{(q)}_{h_q(i)} w^{-a_q sigma_q i} / W(-o_q(i)); lower median; 0 when no hashing qualifies.
// e_q of candidate i under one hashing (sigma, b, a) with bins u; false where the window gain is too small
__device__ __forceinline__ bool estimate_term(uint32_t i, uint32_t sigma, uint32_t b, uint32_t a, const double2* u,
                                              uint32_t n, uint32_t nmask, uint32_t logNp, const double* wtab, double gmin,
                                              const double2* tw, uint32_t tw_shift, double2* e) {
    uint32_t j;
    const int32_t o = gen_offset((sigma * (i - b)) & nmask, n, nmask, logNp, &j);
    const double gain = wtab[o < 0 ? -o : o];
    const double2 w = root_pow_tab((a * sigma * i) & nmask, tw, tw_shift), uj = u[j];
    if (!(gain >= gmin)) return false;
    const double2 v = mul_conj_rn(uj, w);
    *e = make_double2(__ddiv_rn(v.x, gain), __ddiv_rn(v.y, gain));
    return true;
}

// w_i of the caller-bins entry: one thread per candidate, u = nrep x B bins
__device__ double2 estimate_one(uint32_t i, uint32_t nrep, const uint64_t* sig, const uint64_t* bb, const uint64_t* aa,
                                const double2* u, uint32_t B, uint32_t n, uint32_t nmask, uint32_t logNp,
                                const double* wtab, double gmin, const double2* tw, uint32_t tw_shift) {
    double re[kMaxRest], im[kMaxRest];
    uint32_t m = 0;
    for (uint32_t q = 0; q < nrep; ++q) {
        double2 e;
        if (!estimate_term(i, (uint32_t)sig[q], (uint32_t)bb[q], (uint32_t)aa[q], u + (size_t)q * B, n, nmask, logNp, wtab,
                           gmin, tw, tw_shift, &e))
            continue;
        const double x = e.x, y = e.y;
        // insertion into the sorted prefixes
        uint32_t pr = m, pi = m;
        while (pr > 0 && re[pr - 1] > x) {
            re[pr] = re[pr - 1];
            --pr;
        }
        re[pr] = x;
        while (pi > 0 && im[pi - 1] > y) {
            im[pi] = im[pi - 1];
            --pi;
        }
        im[pi] = y;
        ++m;
    }
    if (m == 0) return make_double2(0.0, 0.0);
    return make_double2(re[(m - 1) / 2], im[(m - 1) / 2]);
}

// (mag2 descending, index ascending) order of candidates via a bitonic sort of a permutation over the
// smallest power of two >= m (<= P).  mag2 >= 0 is finite, so its IEEE bit pattern orders like its
// value and the comparisons run on the integer units (GB300's FP64 pipe runs at 1/64 rate).
__device__ void sort_by_magnitude(const double* mag, const uint32_t* idx, uint32_t m, uint32_t P, uint32_t* perm) {
    uint32_t Pm = 1;
    while (Pm < m && Pm < P) Pm <<= 1;
    for (uint32_t p = threadIdx.x; p < Pm; p += kThreads) perm[p] = p;
    __syncthreads();
    const unsigned long long* mb = reinterpret_cast<const unsigned long long*>(mag);
    auto before = [&](uint32_t a, uint32_t b) -> bool {  // a ranks before b
        if (a >= m) return false;
        if (b >= m) return true;
        const unsigned long long x = mb[a], y = mb[b];
        if (x != y) return x > y;
        return idx[a] < idx[b];
    };
    for (uint32_t k = 2; k <= Pm; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = threadIdx.x; i < Pm; i += kThreads) {
                const uint32_t ixj = i ^ j;
                if (ixj > i) {
                    const bool up = (i & k) == 0;
                    const uint32_t pa = perm[i], pb = perm[ixj];
                    const bool swap = up ? before(pb, pa) : before(pa, pb);
                    if (swap) {
                        perm[i] = pb;
                        perm[ixj] = pa;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------------------------------------
// 3. LocateSignal and EstimateValues per bin
// ------------------------------------------------------------------------------------------------
// LocateSignal with t threads per bin (in one warp), thread q owning subregion q: a CTA holds
// kThreads / t bins of one request (the bins are independent until L is formed).  The phases and betas
// of every level are brought to shared memory at once, so the levels follow one another without a
// barrier: a level is R_loc vote tests per thread, one 64-bit product each, and a decision by ballots
// and shuffles inside the bin's lanes (that of locate_bin_t, on the same integers).  The candidate of
// bin j (pi^{-1} of the integer nearest the centre of its last region, kNoIndex for bottom) goes to
// L[s B + j].  EstimateValues' R_est divisions per candidate then spread over the CTA (one
// (candidate, hashing) per thread: GB300 issues FP64 at 1/64 of the FP32 rate, so the estimates of a
// request run on as many SMs as its bins do), and two threads per candidate sort the quotients for
// the medians.  Bound by latency: the level chain, then one chain of FP64 operations.
//
// A vote compares the position e / M of beta (m + sigma b) with the arc of half width s / 2 around c_j,
// both as 32-bit fractions of a turn: with M = n 2^F scaled to 2^64 the product wraps by itself and its
// upper word is the position.  The pipeline's c_j comes from an FP32 arctangent of the product
// u_j conj(u'_j) (in FP64, or good to 2^-46): rounding it to float (see direction) and atan2f's few-ulp error
// move it by less than 2e-7 of a turn, and the 32-bit fractions by less than 1e-9.  A vote within 2^-20 of a turn (about 1e-6) of an
// arc end is decided by the FP64 test on the FP64 phase of the pair's stored bins; every other one is
// farther than that error from the arc ends of either phase, so both give the same vote.
constexpr int kLocBins = kThreads / 8;               // bins per CTA at the smallest t
constexpr uint32_t kPhaseGuard = (1u << 12) + 8u;    // 2^-20 of a turn, and the fractions' own rounding
struct LocLayout {
    size_t beta, vx, vy, c, ok, total;
};
__host__ __device__ inline LocLayout loc_layout(uint32_t npairs, uint32_t nb, uint32_t R_est) {
    LocLayout L;
    size_t off = 0;
    L.beta = smem_take(&off, (size_t)npairs * 8);
    L.vx = smem_take(&off, (size_t)nb * R_est * 8);
    L.vy = smem_take(&off, (size_t)nb * R_est * 8);
    L.c = smem_take(&off, (size_t)npairs * nb * 4);
    L.ok = smem_take(&off, (size_t)nb * R_est * 4);
    L.total = off;
    return L;
}
size_t general_locate_smem(uint32_t npairs, uint32_t t, uint32_t R_est) {
    return loc_layout(npairs, kThreads / t, R_est).total;
}

__global__ void __launch_bounds__(kThreads) k_gen_locate(const GenArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_cand[kLocBins], s_draw[3][kMaxRest];  // candidates; sigma, b, a of the estimation hashings
    __shared__ double s_med[2][kLocBins];
    const uint32_t s = a.req_base + blockIdx.y, tid = threadIdx.x;
    const uint32_t t = a.t;  // 8, 16 or 32 (the schedule checks it)
    const uint32_t q = tid & (t - 1), lb = tid / t, nb = kThreads / t;
    const uint32_t B = a.B;
    const uint32_t j0 = blockIdx.x * nb, j = j0 + lb;
    const LocLayout Ly = loc_layout(a.npairs, nb, a.R_est);
    uint64_t* s_beta = reinterpret_cast<uint64_t*>(smem + Ly.beta);
    uint32_t* s_c = reinterpret_cast<uint32_t*>(smem + Ly.c);  // [npairs][nb]
    const ReqView rq = gen_req(a, s);
    const uint32_t* phase = a.phase + (size_t)s * a.phase_stride;
    for (uint32_t g = tid; g < a.npairs; g += kThreads) {
        const uint32_t D = g / a.R_loc;
        uint32_t aa;
        uint64_t be;
        inner_a_beta(rq.seed, rq.id, a.round, g, a.nmask, a.beta_lo[D], a.beta_hi[D], &aa, &be);
        s_beta[g] = be;
    }
    if (tid >= kThreads - 32 && tid - (kThreads - 32) < a.R_est) {
        const uint32_t e = tid - (kThreads - 32);
        const Words4 w = draw(rq.seed, rq.id, a.round, e, kKindEstimate);
        s_draw[0][e] = (w.w[0] & a.nmask) | 1u;
        s_draw[1][e] = w.w[1] & a.nmask;
        s_draw[2][e] = w.w[2] & a.nmask;
    }
    uint32_t sigma, b;
    locate_sigma_b(rq.seed, rq.id, a.round, a.nmask, &sigma, &b);
    const uint64_t n = a.n, Np = n >> a.logB;
    const uint32_t logM = (uint32_t)(63 - __clzll((long long)n)) + kFracBits;
    const uint64_t M = uint64_t(1) << logM, mask = M - 1;
    const uint32_t sh = 64u - logM;
    const uint64_t sb_fp = ((uint64_t)((sigma * b) & a.nmask)) << kFracBits;
    // half width of the vote arc, s / 2 of a turn (s = 1.5 takes every vote, as any larger s does)
    const uint32_t hw = (uint32_t)__double2uint_rn((a.s > 1.5 ? 1.5 : a.s) * 2147483648.0);
    const double2* rbins = a.bins + (size_t)s * a.bins_stride;
    // the bin's region (start l_fp, width w_D) and its bottom flag live in registers, the same in every
    // lane of the bin's group (t divides 32)
    uint64_t l_fp = ((((uint64_t)j * Np) + n - Np / 2) & (n - 1)) << kFracBits;  // centred on the bin
    after_previous(a);
    for (uint32_t i = tid; i < a.npairs * nb; i += kThreads) {
        const uint32_t g = i / nb, bin = j0 + (i & (nb - 1));
        s_c[i] = bin < B ? phase[(size_t)g * B + bin] : 0u;
    }
    bool valid = j < B;
    const uint32_t lane = tid & 31u, gbase = lane & ~(t - 1u);
    const uint32_t gmask = t == 32u ? 0xFFFFFFFFu : ((1u << t) - 1u) << gbase;
    __syncthreads();
    for (uint32_t D = 0; D < a.dmax; ++D) {
        const uint64_t w_fp = (Np << kFracBits) >> ((uint64_t)D * a.logtp);
        const uint64_t half_step = w_fp / (2 * (uint64_t)t), step = w_fp / t;
        uint32_t v = 0;
        if (valid) {
            // m_q = l + (2q - 1) w / 2t (q from 1): this thread's subregion centre, and sigma b
            const uint64_t pos = (l_fp + half_step + sb_fp + (uint64_t)q * step) << sh;
            const uint32_t* cl = s_c + D * a.R_loc * nb + lb;
            const uint64_t* bl = s_beta + D * a.R_loc;
            for (uint32_t r = 0; r < a.R_loc; ++r) {
                const uint64_t e = bl[r] * pos;  // the position times 2^64 / M, mod 2^64
                const int32_t d = (int32_t)((uint32_t)(e >> 32) - cl[r * nb]);
                const uint32_t ad = (uint32_t)(d < 0 ? -(int64_t)d : (int64_t)d);
                bool hit = ad < hw;
                if (ad + kPhaseGuard - hw <= 2u * kPhaseGuard) {
                    const double2* pb = rbins + (size_t)2 * (D * a.R_loc + r) * B;
                    hit = vote_hit_exact(phase01(mul_conj_rn(pb[j], pb[B + j])), e >> sh, M, a.s);
                }
                v += hit ? 1u : 0u;
            }
        }
        // the level's decision (every lane of the warp takes part; a group's lanes share `valid`):
        // Q* nonempty iff some subregion has more than R_loc / 2 votes; then the window of 4
        // consecutive subregions with the most votes, the first on ties, gives the new region
        const bool any = (__ballot_sync(0xFFFFFFFFu, 2u * v > a.R_loc) & gmask) != 0u;
        uint32_t sum = v + __shfl_down_sync(0xFFFFFFFFu, v, 1, (int)t) + __shfl_down_sync(0xFFFFFFFFu, v, 2, (int)t) +
                       __shfl_down_sync(0xFFFFFFFFu, v, 3, (int)t);
        uint32_t key = q + 4u <= t ? (sum << 8) | (255u - q) : 0u;  // larger sum, then smaller q
        for (uint32_t off = t >> 1; off > 0; off >>= 1) key = max(key, __shfl_xor_sync(0xFFFFFFFFu, key, (int)off, (int)t));
        if (valid) {
            if (!any)
                valid = false;
            else
                l_fp = (l_fp + (uint64_t)(255u - (key & 255u)) * step) & mask;
        }
        if (q == 0 && j < B && a.dbg_lfp) {  // trace: the region and flag after this level
            a.dbg_lfp[((size_t)s * a.dmax + D) * B + j] = l_fp;
            a.dbg_valid[((size_t)s * a.dmax + D) * B + j] = (uint8_t)(valid ? 1 : 0);
        }
    }
    if (q == 0) {
        uint32_t cand = kNoIndex;
        if (valid) {
            const uint64_t wlast = (Np << kFracBits) >> ((uint64_t)a.dmax * a.logtp);
            const uint32_t tau = (uint32_t)(((l_fp + wlast / 2 + (1ull << (kFracBits - 1))) >> kFracBits) & (n - 1));
            cand = ((inverse_odd(sigma) & a.nmask) * tau + b) & a.nmask;
        }
        s_cand[lb] = cand;
        if (j < B) a.L[(size_t)s * B + j] = cand;
    }
    __syncthreads();
    // EstimateValues: e_q of every (candidate, hashing)
    double* vx = reinterpret_cast<double*>(smem + Ly.vx);
    double* vy = reinterpret_cast<double*>(smem + Ly.vy);
    uint32_t* ok = reinterpret_cast<uint32_t*>(smem + Ly.ok);
    const double2* ebins = rbins + (size_t)2 * a.npairs * B;
    const uint32_t logNp = logM - kFracBits - a.logB;
    for (uint32_t i = tid; i < nb * a.R_est; i += kThreads) {
        const uint32_t bin = i & (nb - 1), h = i / nb, c = s_cand[bin];
        double2 e = make_double2(0.0, 0.0);
        bool good = false;
        if (c != kNoIndex)
            good = estimate_term(c, s_draw[0][h], s_draw[1][h], s_draw[2][h], ebins + (size_t)h * B, (uint32_t)n, a.nmask,
                                 logNp, a.wtab, a.est_gmin, a.tw, a.tw_shift, &e);
        vx[i] = e.x;
        vy[i] = e.y;
        ok[i] = good ? 1u : 0u;
    }
    __syncthreads();
    // medians: thread (bin, component) sorts its quotients in place, in hashing order
    if (tid < 2 * nb) {
        const uint32_t bin = tid & (nb - 1);
        double* v = tid < nb ? vx : vy;
        uint32_t m = 0;
        for (uint32_t h = 0; h < a.R_est; ++h) {
            if (!ok[h * nb + bin]) continue;
            const double x = v[h * nb + bin];
            uint32_t p = m;
            while (p > 0 && v[(p - 1) * nb + bin] > x) {
                v[p * nb + bin] = v[(p - 1) * nb + bin];
                --p;
            }
            v[p * nb + bin] = x;
            ++m;
        }
        s_med[tid < nb ? 0 : 1][bin] = m == 0 ? 0.0 : v[((m - 1) / 2) * nb + bin];
    }
    __syncthreads();
    if (tid < nb && j0 + tid < B && s_cand[tid] != kNoIndex) {
        const double2 w = make_double2(s_med[0][tid], s_med[1][tid]);
        a.est_w[(size_t)s * B + j0 + tid] = w;
        a.est_mag[(size_t)s * B + j0 + tid] = __dadd_rn(__dmul_rn(w.x, w.x), __dmul_rn(w.y, w.y));
    }
}

// ------------------------------------------------------------------------------------------------
// 4. top k' of the distinct candidates, zhat += w_J
// ------------------------------------------------------------------------------------------------
// One CTA per request.  Bins that decoded the same frequency are reduced to one (a hash table in shared
// memory: copies carry the same estimate, so which one stays does not matter), the k' first in the
// order (magnitude descending, index ascending) are found by a radix selection on the bits of
// (mag2, ~index) -- mag2 >= 0, so its IEEE pattern orders like its value, on the integer units -- and
// only those are sorted by index, for the merge with zhat.  Bound by latency: about 30 barriers.
constexpr uint32_t kSelThreads = 1024;
constexpr uint32_t kSelDigits = 1024;  // one digit value per thread
struct SelLayout {
    size_t table, js, zi, dup, total;
    uint32_t H, P;
};
__host__ __device__ inline SelLayout sel_layout(uint32_t B, uint32_t kprime, uint32_t zcap) {
    SelLayout L;
    size_t off = 0;
    L.H = 2;
    while (L.H < 2 * B) L.H <<= 1;
    const uint32_t nJ = kprime < B ? kprime : B;
    L.P = 2;
    while (L.P < nJ) L.P <<= 1;
    L.table = smem_take(&off, (size_t)L.H * 4);
    L.js = smem_take(&off, (size_t)L.P * 8);
    L.zi = smem_take(&off, (size_t)zcap * 4);
    L.dup = smem_take(&off, (size_t)L.P * 4);
    L.total = off;
    return L;
}
size_t general_select_smem(uint32_t B, uint32_t kprime, uint32_t zcap) { return sel_layout(B, kprime, zcap).total; }

// exclusive prefix sum over the CTA of one value per thread; tmp holds 33 words.  Starts and ends with
// every thread done with tmp.
__device__ __forceinline__ uint32_t sel_scan(uint32_t v, uint32_t* tmp, uint32_t* total) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (uint32_t off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = tmp[lane];
        uint32_t wi = w;
#pragma unroll
        for (uint32_t off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += y;
        }
        tmp[lane] = wi - w;
        if (lane == 31) tmp[32] = wi;
    }
    __syncthreads();
    const uint32_t r = tmp[warp] + incl - v;
    *total = tmp[32];
    __syncthreads();
    return r;
}

// Ascending sort of the nJ distinct keys js[0..nJ) (js holds P >= nJ words, P a power of two).
__device__ __forceinline__ void sel_sort(unsigned long long* js, uint32_t nJ) {
    const uint32_t tid = threadIdx.x;
    uint32_t P = 2;
    while (P < nJ) P <<= 1;
    if (P <= kSelThreads) {  // one key per thread; partners less than 32 apart are exchanged by shuffles
        unsigned long long k = tid < nJ ? js[tid] : ~0ull;
        for (uint32_t size = 2; size <= P; size <<= 1) {
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                unsigned long long o;
                if (stride < 32) {
                    o = __shfl_xor_sync(0xffffffffu, k, (int)stride);
                } else {
                    __syncthreads();
                    if (tid < P) js[tid] = k;
                    __syncthreads();
                    o = tid < P ? js[tid ^ stride] : k;
                }
                const bool up = (tid & size) == 0, lower = (tid & stride) == 0;
                if ((lower == up) == (o < k)) k = o;
            }
        }
        __syncthreads();
        if (tid < nJ) js[tid] = k;
        __syncthreads();
        return;
    }
    for (uint32_t p = nJ + tid; p < P; p += kSelThreads) js[p] = ~0ull;
    __syncthreads();
    for (uint32_t size = 2; size <= P; size <<= 1)
        for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
            for (uint32_t i = tid; i < P; i += kSelThreads) {
                const uint32_t o = i ^ stride;
                if (o > i) {
                    const unsigned long long x = js[i], y = js[o];
                    if ((i & size) == 0 ? x > y : x < y) {
                        js[i] = y;
                        js[o] = x;
                    }
                }
            }
            __syncthreads();
        }
}

// PER: bins per thread (B <= PER kSelThreads)
template <int PER>
__global__ void __launch_bounds__(kSelThreads) k_gen_select(const GenArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t hist[kSelDigits], tmp[33], s_digit, s_above, s_in;
    const uint32_t s = a.req_base + blockIdx.x, tid = threadIdx.x, B = a.B, lane = tid & 31u;
    const SelLayout Ly = sel_layout(B, a.kprime, a.zcap);
    uint32_t* table = reinterpret_cast<uint32_t*>(smem + Ly.table);
    unsigned long long* js = reinterpret_cast<unsigned long long*>(smem + Ly.js);  // (index, bin) of J
    uint32_t* zs = reinterpret_cast<uint32_t*>(smem + Ly.zi);
    uint32_t* dup = reinterpret_cast<uint32_t*>(smem + Ly.dup);
    uint32_t* zi = a.zidx + (size_t)s * a.zcap;
    double2* zv = a.zval + (size_t)s * a.zcap;
    const double2* ew = a.est_w + (size_t)s * B;
    for (uint32_t h = tid; h < Ly.H; h += kSelThreads) table[h] = kNoIndex;
    hist[tid] = 0;
    after_previous(a);
    // the candidates, and zhat's indices for the merge
    uint32_t cand[PER];
    unsigned long long mag[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint32_t j = tid + (uint32_t)i * kSelThreads;
        cand[i] = j < B ? a.L[(size_t)s * B + j] : kNoIndex;
        mag[i] = j < B ? reinterpret_cast<const unsigned long long*>(a.est_mag)[(size_t)s * B + j] : 0ull;
    }
    const uint32_t nz = min(a.zcount[s], a.zcap);
    for (uint32_t e = tid; e < nz; e += kSelThreads) zs[e] = zi[e];
    __syncthreads();
    // L without repetitions: the first to claim an index keeps it (at most B of H >= 2 B places taken)
    uint32_t state = 0, kept = 0;  // bit i: candidate i still undecided; in J
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        if (cand[i] == kNoIndex) continue;
        uint32_t h = (cand[i] * 2654435769u) >> (__clz((int)Ly.H) + 1);  // the product's top log2 H bits
        for (;;) {
            const uint32_t old = atomicCAS(&table[h], kNoIndex, cand[i]);
            if (old == kNoIndex) {
                state |= 1u << i;
                break;
            }
            if (old == cand[i]) break;
            h = (h + 1) & (Ly.H - 1);
        }
    }
    uint32_t nL;
    sel_scan((uint32_t)__popc((int)state), tmp, &nL);
    // J: the k' first by (mag2 descending, index ascending).  Digits of 10 bits from the top of the key
    // (mag2, ~index); a digit's histogram over the undecided candidates tells which value holds the
    // k'-th, those above it are in J, those below are not
    if (nL <= a.kprime) {
        kept = state;
    } else {
        uint32_t need = a.kprime;
        for (uint32_t pass = 0;; ++pass) {
            uint32_t dg[PER];
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                // 64 bits of mag2 as 6 x 10 + 4, then 32 of ~index as 3 x 10 + 2
                if (pass < 7)
                    dg[i] = pass < 6 ? (uint32_t)(mag[i] >> (54 - 10 * pass)) & 1023u : (uint32_t)mag[i] & 15u;
                else
                    dg[i] = pass < 10 ? (~cand[i] >> (22 - 10 * (pass - 7))) & 1023u : ~cand[i] & 3u;
                const bool in = (state >> i) & 1u;
                const unsigned act = __ballot_sync(0xffffffffu, in);
                if (in) {  // one shared-memory atomic per digit value and warp
                    const unsigned same = __match_any_sync(act, dg[i]);
                    if (lane == (uint32_t)__ffs((int)same) - 1u) atomicAdd(&hist[dg[i]], (uint32_t)__popc((int)same));
                }
            }
            __syncthreads();
            const uint32_t d = kSelDigits - 1 - tid, c = hist[d];
            uint32_t tot;
            const uint32_t above = sel_scan(c, tmp, &tot);
            hist[d] = 0;  // for the next pass
            if (above < need && need <= above + c) {
                s_digit = d;
                s_above = above;
                s_in = c;
            }
            __syncthreads();
            const uint32_t digit = s_digit;
            const bool all = s_in == need - s_above;  // the whole digit value belongs to J
            need -= s_above;
#pragma unroll
            for (int i = 0; i < PER; ++i)
                if ((state >> i) & 1u) {
                    if (dg[i] > digit || (all && dg[i] == digit)) kept |= 1u << i;
                    if (dg[i] != digit || all) state &= ~(1u << i);
                }
            if (all) break;  // the keys are distinct, so the last digit at the latest ends it
            __syncthreads();  // s_digit, s_above, s_in are rewritten by the next pass
        }
    }
    uint32_t nJ;
    uint32_t at = sel_scan((uint32_t)__popc((int)kept), tmp, &nJ);
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if ((kept >> i) & 1u) js[at++] = ((unsigned long long)cand[i] << 32) | (tid + (uint32_t)i * kSelThreads);
    __syncthreads();
    sel_sort(js, nJ);
    // zhat <- zhat + w_J; nothing is dropped in the general case.  An entry of J already in zhat is added
    // to it (zhat first); the others go to c - (repeated ones before c) + (zhat entries below)
    auto jidx = [&](uint32_t c) { return (uint32_t)(js[c] >> 32); };
    uint32_t ndup = 0;  // J's repeated entries, counted before each
    for (uint32_t c0 = 0; c0 < nJ; c0 += kSelThreads) {
        const uint32_t c = c0 + tid;
        uint32_t rep = 0;
        if (c < nJ) {
            const uint32_t key = jidx(c), ub = upper_bound_u32(zs, nz, key);
            rep = ub > 0 && zs[ub - 1] == key ? 1u : 0u;
        }
        uint32_t tot;
        const uint32_t before = sel_scan(rep, tmp, &tot);
        if (c < nJ) dup[c] = (ndup + before) | (rep << 31);
        ndup += tot;
    }
    __syncthreads();
    const bool last = a.last_round != 0;
    const uint32_t newcount = nz + nJ - ndup;
    auto put = [&](uint32_t pos, uint32_t key, double2 v) {
        if (pos < a.zcap) {
            zi[pos] = key;
            zv[pos] = v;
        }
        if (last && pos < a.out_cap) {
            a.out_idx[(size_t)s * a.out_cap + pos] = key;
            a.out_val[(size_t)s * a.out_cap + pos] = v;
        }
    };
    // zhat moves up in place: each pass of kSelThreads entries from the top is read before it is
    // written, and writes only at or above the places it read
    for (uint32_t done = 0; done < nz; done += kSelThreads) {
        const uint32_t e = nz - 1 - done - tid;
        const bool mine = done + tid < nz;
        uint32_t key = 0, pos = 0;
        double2 v = make_double2(0.0, 0.0);
        if (mine) {
            key = zs[e];
            v = zv[e];
            uint32_t lo = 0, hi = nJ;  // entries of J below key
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (jidx(mid) < key) lo = mid + 1; else hi = mid;
            }
            const uint32_t d = lo < nJ ? dup[lo] : ndup;
            pos = e + lo - (d & 0x7FFFFFFFu);
            if (lo < nJ && jidx(lo) == key) {
                const double2 w = ew[(uint32_t)js[lo]];
                v = make_double2(v.x + w.x, v.y + w.y);
            }
        }
        __syncthreads();
        if (mine) put(pos, key, v);
    }
    for (uint32_t c = tid; c < nJ; c += kSelThreads) {
        const uint32_t d = dup[c];
        if (d >> 31) continue;
        const uint32_t key = jidx(c);
        put(c - d + upper_bound_u32(zs, nz, key), key, ew[(uint32_t)js[c]]);
    }
    if (tid == 0) {
        const bool overflow = newcount > a.zcap;
        if (overflow) a.zflag[s] = 1;
        a.zcount[s] = overflow ? a.zcap : newcount;
        if (last) {
            const uint32_t count = overflow ? a.zcap : newcount;
            a.out_count[s] = count < a.out_cap ? count : a.out_cap;
            a.out_flag[s] = (a.zflag[s] || count > a.out_cap) ? SFFT_ERR_CAPACITY : SFFT_OK;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// single-step kernels on caller bins
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_locate_votes(const VoteArgs a) {
    const uint32_t logM = (uint32_t)(63 - __clzll((long long)a.n)) + kFracBits;
    const int64_t hw_fix = vote_halfwidth(a.s, logM);
    const uint64_t sb_fp = ((uint64_t)((a.sigma * a.b) & a.nmask)) << kFracBits;
    for (uint32_t j = threadIdx.x; j < a.B; j += kThreads) {
        for (uint32_t q = 0; q < a.t; ++q) a.votes[(size_t)j * a.t + q] = 0;
        if (!a.valid[j]) continue;
        uint64_t l = a.l_fp[j];
        uint8_t v = 1;
        locate_bin(a.t, a.nrep, a.beta,
                   [&](uint32_t r) {
                       return phase01(mul_conj_rn(a.u[(size_t)r * a.B + j], a.up[(size_t)r * a.B + j]));
                   },
                   sb_fp, a.w_fp, logM, a.s, hw_fix, l, v, a.votes + (size_t)j * a.t);
        a.l_fp[j] = l;
        a.valid[j] = v;
    }
}

struct EstLayout {
    size_t w, mag, perm, keep, scan, total;
    uint32_t P;
};
__host__ __device__ inline EstLayout est_layout(uint32_t m) {
    EstLayout L;
    size_t off = 0;
    uint32_t P = 1;
    while (P < m) P <<= 1;
    L.P = P;
    L.w = smem_take(&off, (size_t)m * 16);
    L.mag = smem_take(&off, (size_t)m * 8);
    L.perm = smem_take(&off, (size_t)P * 4);
    L.keep = smem_take(&off, (size_t)m * 4);
    L.scan = smem_take(&off, (size_t)(kThreads + 8) * 4);
    L.total = off;
    return L;
}

__global__ void __launch_bounds__(kThreads) k_estimate_from_bins(const EstArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t tid = threadIdx.x;
    const EstLayout Ly = est_layout(a.nL > 0 ? a.nL : 1);
    double2* wv = reinterpret_cast<double2*>(smem + Ly.w);
    double* mag = reinterpret_cast<double*>(smem + Ly.mag);
    uint32_t* perm = reinterpret_cast<uint32_t*>(smem + Ly.perm);
    uint32_t* keep = reinterpret_cast<uint32_t*>(smem + Ly.keep);
    uint32_t* scan = reinterpret_cast<uint32_t*>(smem + Ly.scan);
    const uint32_t logNp = (uint32_t)(63 - __clzll((long long)a.n)) - a.logB;
    for (uint32_t c = tid; c < a.nL; c += kThreads) {
        const double2 w = estimate_one(a.L[c], a.nrep, a.sig, a.bb, a.aa, a.u, a.B, (uint32_t)a.n, a.nmask, logNp, a.wtab,
                                       a.est_gmin, a.tw, a.tw_shift);
        wv[c] = w;
        mag[c] = __dadd_rn(__dmul_rn(w.x, w.x), __dmul_rn(w.y, w.y));
    }
    __syncthreads();
    sort_by_magnitude(mag, a.L, a.nL, Ly.P, perm);
    const uint32_t nJ = a.nL < a.kprime ? a.nL : a.kprime;
    for (uint32_t c = tid; c < a.nL; c += kThreads) keep[c] = 0;
    __syncthreads();
    for (uint32_t r = tid; r < nJ; r += kThreads) keep[perm[r]] = 1;
    __syncthreads();
    const uint32_t total = block_exclusive_scan(keep, a.nL, scan);
    for (uint32_t c = tid; c < a.nL; c += kThreads) {
        const uint32_t nxt = c + 1 < a.nL ? keep[c + 1] : total;
        if (nxt != keep[c]) {
            a.widx[keep[c]] = a.L[c];
            a.wval[keep[c]] = wv[c];
        }
    }
    if (tid == 0) *a.count = total;
}

// ------------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------------
static cudaError_t raise_smem(const void* kernel, size_t bytes, size_t* lim) {
    if (bytes <= *lim) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) *lim = bytes;
    return e;
}
cudaError_t general_set_smem(size_t finish, size_t locate, size_t select, size_t estimate) {
    static std::mutex mu;  // plans may be created from several threads
    std::lock_guard<std::mutex> lk(mu);
    static size_t lim[6] = {0, 0, 0, 0, 0, 0};
    cudaError_t e = raise_smem((const void*)k_gen_finish, finish, &lim[0]);
    if (e == cudaSuccess) e = raise_smem((const void*)k_gen_locate, locate, &lim[1]);
    if (e == cudaSuccess) e = raise_smem((const void*)k_gen_select<1>, select, &lim[2]);
    if (e == cudaSuccess) e = raise_smem((const void*)k_gen_select<2>, select, &lim[3]);
    if (e == cudaSuccess) e = raise_smem((const void*)k_gen_select<4>, select, &lim[4]);
    if (e == cudaSuccess) e = raise_smem((const void*)k_estimate_from_bins, estimate, &lim[5]);
    return e;
}

// a launch that may overlap the end of the one before it (see after_previous)
template <typename Arg>
static cudaError_t launch_after(void (*kernel)(Arg), dim3 grid, uint32_t threads, size_t smem, cudaStream_t st, const Arg& arg) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, arg);
}

constexpr uint32_t kGatherPlaces = 2 * 152;  // CTAs of k_gen_gather the chip holds
// pairs per CTA: as many as leave the chip two waves of CTAs over the whole call's `batch` requests, so that a
// tap's window product serves more hashings
static uint32_t gather_blocks(const GeneralRound& g) { return g.B > (uint32_t)kThreads ? g.B / kThreads : 1u; }
static uint32_t gather_pairs_per_cta(const GeneralRound& g, uint32_t batch) {
    const uint64_t pairs = (uint64_t)gather_blocks(g) * g.npairs * batch;
    return pairs >= 8 * kGatherPlaces ? 4u : (pairs >= 4 * kGatherPlaces ? 2u : 1u);
}
// a round's CTAs per request
static uint32_t gather_ctas(const GeneralRound& g, uint32_t R_est, uint32_t P) {
    return gather_blocks(g) * (R_est + (g.npairs + P - 1) / P);
}

// Whether the kernels of a call start early (after_previous): where the call's gathers all have a place on the
// chip.  CTAs that only wait hold places: at n = 2^20, k = 500 (about 1000 CTAs a request) one request took
// 348 us with early starts and 305 without, n = 2^18, k = 50, batch 4 (724) 168 and 155, n = 2^16, k = 8,
// batch 8 (808) 98 and 85; where they fit, early starts gave n = 2^16, k = 8, batch 3 70.5 us against 72.2,
// n = 2^18, k = 50, one request 108.0 against 108.6.
bool general_early(const GeneralRound* g, uint32_t R, uint32_t R_est, uint32_t batch) {
    uint64_t ctas = 0;
    for (uint32_t r = 0; r < R; ++r) ctas += (uint64_t)gather_ctas(g[r], R_est, gather_pairs_per_cta(g[r], batch)) * batch;
    return ctas <= kGatherPlaces;
}

template <int NR>
static cudaError_t launch_gather_nr(const GenArgs* a, const GeneralRound* g, uint32_t R, uint32_t batch, cudaStream_t st) {
    GatherParams<NR> gp;
    gp.R = R;
    gp.seg[0] = 0;
    for (uint32_t r = 0; r < R; ++r) {
        gp.P[r] = gather_pairs_per_cta(g[r], a[r].batch);
        gp.seg[r + 1] = gp.seg[r] + gather_ctas(g[r], a[r].R_est, gp.P[r]);
        gp.r[r] = a[r];
    }
    return launch_after<const GatherParams<NR>>(k_gen_gather<NR>, dim3(gp.seg[R], batch), kThreads, 0, st, gp);
}

cudaError_t launch_general_gather(const GenArgs* a, const GeneralRound* g, uint32_t R, uint32_t batch, cudaStream_t st) {
    if (R == 0 || R > kMaxGenRounds) return cudaErrorInvalidValue;
    for (uint32_t r = 0; r < R; ++r)
        if (g[r].perm) {
            const uint64_t per = (uint64_t)kThreads * 8, blocks = (a[r].n + per - 1) / per;
            k_gen_permute<<<dim3((uint32_t)(blocks < 65535 ? blocks : 65535), batch), kThreads, 0, st>>>(a[r]);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    return R <= 6 ? launch_gather_nr<6>(a, g, R, batch, st) : launch_gather_nr<kMaxGenRounds>(a, g, R, batch, st);
}

cudaError_t launch_general_round(const GenArgs& a, uint32_t batch, const GeneralRound& r, cudaStream_t st) {
    using Arg = const GenArgs;
    cudaError_t e = launch_after<Arg>(k_gen_finish, dim3(r.ngroups, batch), kThreads, r.smem_finish, st, a);
    if (e != cudaSuccess) return e;
    const uint32_t nb = kThreads / r.t;  // bins per CTA
    e = launch_after<Arg>(k_gen_locate, dim3((r.B + nb - 1) / nb, batch), kThreads, r.smem_locate, st, a);
    if (e != cudaSuccess) return e;
    return launch_after<Arg>(r.B <= kSelThreads ? k_gen_select<1> : (r.B <= 2 * kSelThreads ? k_gen_select<2> : k_gen_select<4>),
                             dim3(batch), kSelThreads, r.smem_select, st, a);
}

cudaError_t launch_locate_votes(const VoteArgs& a, cudaStream_t st) {
    k_locate_votes<<<1, kThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_estimate_from_bins(const EstArgs& a, cudaStream_t st) {
    const size_t smem = est_layout(a.nL > 0 ? a.nL : 1).total;
    cudaError_t e = general_set_smem(0, 0, 0, smem);
    if (e != cudaSuccess) return e;
    k_estimate_from_bins<<<1, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace sfft
