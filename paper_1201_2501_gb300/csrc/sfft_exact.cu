// sfft_exact.cu -- the exact-mode sparse FFT on sm_103a (Algorithm 1 of Hassanieh, Indyk, Katabi,
// Price) for a whole batch of requests.
//
// Work unit: one chunk (by default 2048 consecutive window taps) of one round of one request.  Its
// CTA performs steps 1-2 of HashToBins (proof of Lemma "hashtobins") for all hashings of the round
// (a = 0 and the ladder shifts share one staged run of samples, since x_{sigma(t - beta)} is sample
// t - beta of the sigma-strided sequence): it gathers the permuted samples, applies window and
// modulation, folds them modulo B and stores the partial fold.  The last arrival of a request's round
// (arrival counter, no waiting) sums the partials in chunk order, runs the B-point FFTs (step 3),
// subtracts the recovered coefficients in FP64 (step 4), decodes locations and values
// (NoiselessSparseFFTInner's loop over J) and merges the result into zhat (NoiselessSparseFFT).
//
// k_exact_step runs every round of the batch in one launch: the sample positions of all rounds are
// known up front (sigma, b come from the counter-based draws, never from zhat), so all chunks are
// gathered at once and only the finishers are ordered, round t's by the arrival of round t - 1's.
// k_exact_batch does the same for requests of different plans; k_exact_round runs one round (the
// single-hashing entry points).  Every reduction has a fixed order and no floating-point atomics exist, so results are
// bit-reproducible.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <type_traits>
#include <stdint.h>

#include "philox.cuh"
#include "sfft_device.cuh"
#include "sfft_internal.h"

namespace sfft {

template <typename R>
__device__ __forceinline__ const R* taps_of(const ExactArgs& a);
template <>
__device__ __forceinline__ const float* taps_of<float>(const ExactArgs& a) {
    return a.taps32;
}
template <>
__device__ __forceinline__ const double* taps_of<double>(const ExactArgs& a) {
    return a.taps64;
}

static_assert(kThreads / kOwnerRes >= kMaxHash, "a thread per (residue, hashing)");
// samples in flight per thread of gather_owner
template <typename R>
__host__ __device__ constexpr uint32_t owner_loads() {
    return sizeof(R) == sizeof(float) ? 16 : 8;
}

// ------------------------------------------------------------------------------------------------
// shared-memory layout of the finishing phase
// ------------------------------------------------------------------------------------------------
struct FinLayout {
    size_t U, ent_idx, ent_bin, ent_val, ent_gain, ent_sub, ent_sub_f, mask, bin_cnt, bin_start, bin_list, cand_idx, cand_val, srt_idx, srt_val, out_idx, out_val, keep, scan;
    size_t total;
};
// masks: the entries of each bin as bits (the transform's decode), instead of as lists
__host__ __device__ inline FinLayout fin_layout(uint32_t B, uint32_t H, uint32_t zcap, uint32_t csize, bool masks = false) {
    FinLayout L;
    size_t off = 0;
    L.U = smem_take(&off, (size_t)H * B * csize);
    L.ent_idx = smem_take(&off, (size_t)zcap * 4);
    L.ent_bin = smem_take(&off, (size_t)zcap * 4);
    L.ent_val = smem_take(&off, (size_t)zcap * 16);
    L.ent_gain = smem_take(&off, (size_t)zcap * 8);
    L.ent_sub = smem_take(&off, (size_t)zcap * H * 16);
    L.ent_sub_f = smem_take(&off, csize == 8 ? (size_t)zcap * H * 8 : 0);  // FP32 data path
    L.mask = smem_take(&off, masks ? (size_t)B * ((zcap + 31) / 32) * 4 : 0);
    L.bin_cnt = smem_take(&off, masks ? 0 : (size_t)(B + 1) * 4);
    L.bin_start = smem_take(&off, masks ? 0 : (size_t)(B + 1) * 4);
    L.bin_list = smem_take(&off, masks ? 0 : (size_t)zcap * 4);
    L.cand_idx = smem_take(&off, (size_t)B * 4);
    L.cand_val = smem_take(&off, (size_t)B * 16);
    L.srt_idx = smem_take(&off, (size_t)B * 4);
    L.srt_val = smem_take(&off, (size_t)B * 16);
    L.out_idx = smem_take(&off, (size_t)(zcap + B) * 4);
    L.out_val = smem_take(&off, (size_t)(zcap + B) * 16);
    L.keep = smem_take(&off, (size_t)(zcap + B) * 4);
    L.scan = smem_take(&off, (size_t)(kThreads + 8) * 4);
    L.total = off;
    return L;
}

size_t exact_finish_smem(uint32_t B, uint32_t H, uint32_t zcap, bool fp64) {
    return fin_layout(B, H, zcap, fp64 ? 16 : 8).total;
}
size_t exact_decode_smem(uint32_t B, uint32_t H, uint32_t zcap, bool fp64) {
    return fin_layout(B, H, zcap, fp64 ? 16 : 8, true).total;
}
// What the bounds on a plan's arrays count beyond them: 12 bytes a bin for a decode by lists, 8 an entry and
// hashing for FP64, arrays of earlier forms.  The bounds (kFinSmemMax, the refusal above 200 KB) were measured
// with these, and a plan keeps its decode, or its refusal.
size_t exact_finish_bound(uint32_t B, uint32_t H, uint32_t zcap, bool fp64) {
    return exact_finish_smem(B, H, zcap, fp64) + (size_t)B * 12 + (fp64 ? (size_t)zcap * H * 8 : 0);
}
size_t exact_decode_bound(uint32_t B, uint32_t H, uint32_t zcap, bool fp64) {
    return exact_decode_smem(B, H, zcap, fp64) + (fp64 ? (size_t)zcap * H * 8 : 0);
}
size_t exact_gather_smem(uint32_t stage, bool fp64) { return (size_t)stage * (fp64 ? 16 : 8); }
constexpr uint32_t owner_batch(bool fp64) {  // taps of a residue per batch
    return (fp64 ? owner_loads<double>() : owner_loads<float>()) * (kThreads / kOwnerRes);
}
size_t exact_owner_smem(uint32_t ring, bool fp64) {  // samples and factors
    return (size_t)(ring + owner_batch(fp64)) * kOwnerRes * (fp64 ? 16 : 8);
}
// samples gather_owner keeps of a residue: those of a batch and of the longest shift (0: too many)
uint32_t exact_owner_ring(uint64_t maxshift, uint32_t B, bool fp64) {
    uint32_t r = 1;
    while (r < owner_batch(fp64) + maxshift / B) r <<= 1;
    return r <= 2 * owner_batch(fp64) ? r : 0;
}

// g w^e of a tap, w = exp(-2 pi i / n), e = sigma b t (taken mod n): a sincospif in FP32; from the factor
// tables in FP64, whose sincospi took most of the FP64 gather's time.  With the bins' FFT and the
// subtraction terms from the tables and the decisions in guarded FP32 (decode_bin_guarded): n = 2^20,
// k = 64, batch 16: 134 us a call, was 228; n = 2^14, k = 8, one request: 42 us, was 73.
__device__ __forceinline__ float2 tap_factor(const ExactArgs& a, float g, uint32_t ex, float two_over_n) {
    const uint32_t e = ex & a.nmask;
    const int32_t es = e > (a.nmask >> 1) ? (int32_t)((int64_t)e - (int64_t)a.n) : (int32_t)e;
    float sn, cs;
    sincospif((float)es * two_over_n, &sn, &cs);
    return make_float2(g * cs, -g * sn);
}
__device__ __forceinline__ double2 tap_factor(const ExactArgs& a, double g, uint32_t ex, double /*two_over_n*/) {
    const double2 w = root_pow_fine(ex & a.nmask, a.tw, a.tw_shift);
    return make_double2(g * w.x, g * w.y);
}
// w^e of a subtraction term in the precision of the data path
template <typename R>
__device__ __forceinline__ double2 term_root(const ExactArgs& a, uint32_t e) {
    return sizeof(R) == sizeof(float) ? root_pow<float>(e, a.nmask) : root_pow_fine(e, a.tw, a.tw_shift);
}

// ------------------------------------------------------------------------------------------------
// Location and estimation of one bin (NoiselessSparseFFTInner's loop body)
// ------------------------------------------------------------------------------------------------
struct DecodeCtx {
    uint32_t n, nmask, B, Np, logNp, H;
    uint32_t sigma, sigma_inv, b, sb;
    uint32_t shift[kMaxHash];  // ladder shifts beta_l (hashing l + 1)
    uint32_t logR[kMaxHash];   // log2(beta_l / B)
    const double* wtab;
    const double* winv;        // 1 / W(o) beside wtab, or null
    double thr, iso_tol, gmin, ref_lo, ref_hi, ref_tol;
    // the same thresholds for the FP32 decisions (ref_lo_f, ref_hi_f already scaled by thr)
    float thr_f, iso_tol_f, ref_lo_f, ref_hi_f, ref_tol_f, inv_n_f;
};

// bin j = round(p / Np) mod B of permuted position p, and the offset o = p - j Np in (-Np/2, Np/2]
__device__ __forceinline__ int32_t offset_of(uint32_t p, uint32_t Np, uint32_t logNp, uint32_t nmask, uint32_t* jbin) {
    const uint32_t jj = ((p + (Np >> 1)) & nmask) >> logNp;
    const uint32_t dd = (p - jj * Np) & nmask;
    *jbin = jj;
    return dd > (nmask >> 1) ? (int32_t)((int64_t)dd - (int64_t)nmask - 1) : (int32_t)dd;
}
__device__ __forceinline__ int32_t offset_of(uint32_t p, const DecodeCtx& d, uint32_t* jbin) {
    return offset_of(p, d.Np, d.logNp, d.nmask, jbin);
}

// the index part of the decode context: sizes, the hashing (sigma, sigma^-1, b) and the ladder
__device__ void fill_ctx_index(DecodeCtx& d, uint64_t n, uint32_t nmask, uint32_t B, uint32_t logB, uint32_t H,
                               const uint64_t* ladder, uint32_t sigma, uint32_t b) {
    d.n = (uint32_t)n;
    d.nmask = nmask;
    d.B = B;
    d.Np = (uint32_t)(n >> logB);
    d.logNp = ilog2_u32(d.Np);
    d.H = H;
    d.sigma = sigma;
    d.sigma_inv = inverse_odd(sigma) & nmask;
    d.b = b;
    d.sb = (sigma * b) & nmask;
    for (int l = 0; l < kMaxHash; ++l) {
        d.shift[l] = (uint32_t)ladder[l];
        d.logR[l] = ladder[l] >= B ? ilog2_u32((uint32_t)(ladder[l] / B)) : 0u;
    }
    d.inv_n_f = __int_as_float((127 - (int)ilog2_u32(d.n)) << 23);  // 2^-log2 n, exact
}

// decode context of a caller-bins decode: thresholds rounded to FP32 here, values divided by W(o)
__device__ void fill_ctx(DecodeCtx& d, uint64_t n, uint32_t nmask, uint32_t B, uint32_t logB, uint32_t H,
                         const uint64_t* ladder, uint32_t sigma, uint32_t b, const double* wtab, double thr,
                         double iso_tol, double gmin, double ref_lo, double ref_hi, double ref_tol) {
    fill_ctx_index(d, n, nmask, B, logB, H, ladder, sigma, b);
    d.wtab = wtab;
    d.winv = nullptr;
    d.thr = thr;
    d.iso_tol = iso_tol;
    d.gmin = gmin;
    d.ref_lo = ref_lo;
    d.ref_hi = ref_hi;
    d.ref_tol = ref_tol;
    d.thr_f = (float)thr;
    d.iso_tol_f = (float)iso_tol;
    d.ref_lo_f = (float)(ref_lo * thr);
    d.ref_hi_f = (float)(ref_hi * thr);
    d.ref_tol_f = (float)ref_tol;
}

// decode context of a round of the transform: the round block carries the FP32 thresholds (rounded
// on the host, so that no FP64 conversion runs here) and the table of 1 / W(o)
__device__ void fill_ctx_round(DecodeCtx& d, const ExactArgs& a, uint32_t sigma, uint32_t b) {
    uint64_t ladder[kMaxHash];
    for (int l = 0; l < kMaxHash; ++l) ladder[l] = l + 1 < kMaxHash ? a.shift64[l + 1] : 0;
    fill_ctx_index(d, a.n, a.nmask, a.B, a.logB, a.H, ladder, sigma, b);
    d.wtab = a.wtab;
    d.winv = a.winv;
    d.thr = a.thr;
    d.iso_tol = a.iso_tol;
    d.gmin = a.gmin;
    d.ref_lo = a.ref_lo;
    d.ref_hi = a.ref_hi;
    d.ref_tol = a.ref_tol;
    d.thr_f = a.thr_f;
    d.iso_tol_f = a.iso_tol_f;
    d.ref_lo_f = a.ref_lo_f;
    d.ref_hi_f = a.ref_hi_f;
    d.ref_tol_f = a.ref_tol_f;
}

// The zhat entries hashed to a bin, in ascending order of their ids e: each(f) calls f(e) for every one.
// kDirect: ids count from the bin's first place, and a decode is returned before its window gain is read, with
// the signed offset o in *oi, or with the id of the entry a re-estimate corrects.
struct ListEntries {
    static constexpr bool kDirect = false;
    const uint32_t* list;
    uint32_t count;
    __device__ __forceinline__ bool any() const { return count != 0; }
    template <typename F>
    __device__ __forceinline__ void each(F f) const {
        for (uint32_t x = 0; x < count; ++x) f(list[x]);
    }
};
struct RunEntries {
    static constexpr bool kDirect = true;
    uint32_t count;
    __device__ __forceinline__ bool any() const { return count != 0; }
    template <typename F>
    __device__ __forceinline__ void each(F f) const {
        for (uint32_t x = 0; x < count; ++x) f(x);
    }
};
struct MaskEntries {  // bit e mod 32 of words[(e / 32) stride]
    static constexpr bool kDirect = false;
    const uint32_t* words;
    uint32_t stride, nwords;
    __device__ __forceinline__ bool any() const {
        uint32_t m = 0;
        for (uint32_t w = 0; w < nwords; ++w) m |= words[w * stride];
        return m != 0;
    }
    template <typename F>
    __device__ __forceinline__ void each(F f) const {
        for (uint32_t w = 0; w < nwords; ++w)
            for (uint32_t m = words[w * stride]; m != 0; m &= m - 1u) f(w * 32u + (uint32_t)__ffs((int)m) - 1u);
    }
};
__device__ __forceinline__ uint32_t index_at(const DecodeCtx& d, uint32_t j, int32_t o) {
    const uint32_t p = (j * d.Np + (uint32_t)o) & d.nmask;
    return (d.sigma_inv * ((p + d.sb) & d.nmask)) & d.nmask;
}
// Decode of one bin (NoiselessSparseFFTInner's loop body).  u[0..H) are the bin's hashings after the
// subtraction of zhat, in the precision of the data path, `ents` its entries, with indices ent_idx[] and window
// gains ent_gain[].  Returns 0 (nothing), 1 (a decode of J kept) or 2 (a re-estimate of a known entry), with
// the index in *oi and the window gain that divides u_0 in *gout (the caller forms the FP64 value; for a decode
// of the FP32 path *ginv is 1 / gain from the table beside W, else 0, and the caller divides).  *above is set
// when |u_0| > thr.
//
// FP64 bins are decided as FP64 decides them: by decode_bin_guarded where FP32 must agree, else here.  FP32
// bins take every decision (magnitudes, phases, the location ladder, isolation and re-estimation tests) in
// FP32 (decode_bin_fp32): they carry ~1e-6 of rounding, the ladder keeps a tolerance of at least tau_dec per
// level and GB300 issues FP64 at 1/64 of FP32, so FP64 arithmetic there would cost most of the finisher's time
// and change no decision outside a measure-zero band at the thresholds.
template <typename Ents>
__device__ __noinline__ int decode_bin_fp64(const DecodeCtx& d, uint32_t j, const double2* u, const Ents ents, const uint32_t* ent_idx, const double* ent_gain, uint32_t* oi, double* gout,
                               double* ginv, bool* above) {
    const double mag0 = cmag(u[0]);
    *ginv = 0.0;  // the FP64 path divides
    const uint32_t L = d.H - 1;
    *above = false;
    if (!(mag0 > d.thr)) {
        // re-estimation of a known value: exactly one entry of the bin must explain the residual
        if (!ents.any() || !(mag0 > d.ref_lo * d.thr && mag0 <= d.ref_hi * d.thr)) return 0;
        double th[kMaxHash];
        for (uint32_t l = 0; l < L; ++l) {
            if (fabs(cmag(u[l + 1]) - mag0) > 0.25 * mag0) return 0;
            th[l] = phase01(mul_conj(u[0], u[l + 1]));
        }
        uint32_t matches = 0, who = 0;
        double gw = 1.0;
        ents.each([&](uint32_t e) {
            const uint32_t i = ent_idx[e];
            const double gain = ent_gain[e];
            if (!(gain >= d.gmin)) return;
            bool ok = true;
            for (uint32_t l = 0; l < L && ok; ++l) {
                const uint32_t ph = (d.shift[l] * d.sigma * i) & d.nmask;
                double dist = fabs(th[l] - (double)ph / (double)d.n);
                if (dist > 0.5) dist = 1.0 - dist;
                ok = dist * 6.283185307179586476925286766559 < d.ref_tol;
            }
            if (ok) {
                ++matches;
                who = Ents::kDirect ? e : i;
                gw = gain;
            }
        });
        if (matches != 1) return 0;
        *oi = who;
        *gout = gw;
        return 2;
    }
    *above = true;
    // location ladder, coarsest shift first: q = sigma i mod n/B.  Every modulus is a power of two,
    // so mod and division are masks and exact scalings.
    uint32_t logM = d.logNp - d.logR[L - 1];
    const double th = phase01(mul_conj(u[0], u[L]));
    uint64_t c = (uint64_t)(int64_t)floor(th * ldexp(1.0, (int)logM) + 0.5) & ((uint64_t(1) << logM) - 1);
    for (int l = (int)L - 2; l >= 0; --l) {
        const uint32_t logMp = d.logNp - d.logR[l];
        const uint32_t logRatio = logMp - logM;
        const double thl = phase01(mul_conj(u[0], u[l + 1]));
        const double y = thl * ldexp(1.0, (int)logRatio) - ldexp((double)c, -(int)logM);
        const int64_t h = (int64_t)floor(y + 0.5) & (int64_t)((uint64_t(1) << logRatio) - 1);
        c += (uint64_t(1) << logM) * (uint64_t)h;
        logM = logMp;
    }
    const uint32_t q = (uint32_t)c;
    const uint32_t dd = (q + d.Np - (d.sb & (d.Np - 1)) + (d.Np >> 1)) & (d.Np - 1);
    const int32_t o = (int32_t)dd - (int32_t)(d.Np >> 1);
    const uint32_t i = index_at(d, j, o);
    for (uint32_t l = 0; l < L; ++l)
        if (fabs(cmag(u[l + 1]) - mag0) > d.iso_tol * mag0) return 0;
    if (Ents::kDirect) {
        *oi = (uint32_t)o;
        return 1;
    }
    const double gain = d.wtab[o < 0 ? -o : o];
    if (!(gain >= d.gmin)) return 0;
    *oi = i;
    *gout = gain;
    return 1;
}

__device__ __forceinline__ float2 mul_conj_f(float2 a, float2 b) {  // a * conj(b)
    return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// phase(z) / 2 pi in [0, 1)
__device__ __forceinline__ float phase01_f(float2 z) {
    float p = atan2f(z.y, z.x) * 0.159154943091895336f;
    if (p < 0.0f) p += 1.0f;
    if (p >= 1.0f) p -= 1.0f;
    return p;
}
__device__ __forceinline__ float pow2_f(int e) { return __int_as_float((127 + e) << 23); }  // 2^e, |e| < 127

// Every loop over hashings is unrolled to kMaxHash with compile-time indices, so u[] and the
// phases stay in registers.
template <typename Ents>
__device__ __forceinline__ int decode_bin_fp32(const DecodeCtx& d, uint32_t j, const float2* u, const Ents& ents,
                                               const uint32_t* ent_idx, const double* ent_gain,
                                               uint32_t* oi, double* gout, double* ginv, bool* above) {
    const float mag0 = hypotf(u[0].x, u[0].y);
    *ginv = 0.0;
    const uint32_t L = d.H - 1;
    *above = false;
    if (!(mag0 > d.thr_f)) {
        // re-estimation of a known value: exactly one entry of the bin must explain the residual
        if (!ents.any() || !(mag0 > d.ref_lo_f && mag0 <= d.ref_hi_f)) return 0;
        float th[kMaxHash - 1];
#pragma unroll
        for (int l = 0; l < kMaxHash - 1; ++l) {
            th[l] = 0.0f;
            if ((uint32_t)l < L) {
                if (fabsf(hypotf(u[l + 1].x, u[l + 1].y) - mag0) > 0.25f * mag0) return 0;
                th[l] = phase01_f(mul_conj_f(u[0], u[l + 1]));
            }
        }
        uint32_t matches = 0, who = 0;
        double gw = 1.0;
        ents.each([&](uint32_t e) {
            const uint32_t i = ent_idx[e];
            const double gain = ent_gain[e];
            if (!(gain >= d.gmin)) return;
            bool ok = true;
#pragma unroll
            for (int l = 0; l < kMaxHash - 1; ++l) {
                if ((uint32_t)l < L && ok) {
                    const uint32_t ph = (d.shift[l] * d.sigma * i) & d.nmask;
                    float dist = fabsf(th[l] - (float)ph * d.inv_n_f);
                    if (dist > 0.5f) dist = 1.0f - dist;
                    ok = dist * 6.28318530717958648f < d.ref_tol_f;
                }
            }
            if (ok) {
                ++matches;
                who = Ents::kDirect ? e : i;
                gw = gain;
            }
        });
        if (matches != 1) return 0;
        *oi = who;
        *gout = gw;
        return 2;
    }
    *above = true;
    // location ladder, coarsest shift first (as decode_bin_fp64).  Products with powers of two are
    // exact; c < 2^logM <= 2^30 and every rounded quantity fits 32 bits, so the conversions are the
    // 32-bit ones.
    float2 uL = u[1];
    uint32_t logRL = d.logR[0];
#pragma unroll
    for (int l = 2; l < kMaxHash; ++l)
        if ((uint32_t)l == L) {
            uL = u[l];
            logRL = d.logR[l - 1];
        }
    uint32_t logM = d.logNp - logRL;
    const float th = phase01_f(mul_conj_f(u[0], uL));
    uint32_t c = (uint32_t)__float2int_rd(th * pow2_f((int)logM) + 0.5f) & ((1u << logM) - 1u);
#pragma unroll
    for (int l = kMaxHash - 3; l >= 0; --l) {
        if (l > (int)L - 2) continue;
        const uint32_t logMp = d.logNp - d.logR[l];
        const uint32_t logRatio = logMp - logM;
        const float thl = phase01_f(mul_conj_f(u[0], u[l + 1]));
        const float y = thl * pow2_f((int)logRatio) - __uint2float_rn(c) * pow2_f(-(int)logM);
        const uint32_t h = (uint32_t)__float2int_rd(y + 0.5f) & ((1u << logRatio) - 1u);
        c += h << logM;
        logM = logMp;
    }
    const uint32_t q = c;
    const uint32_t dd = (q + d.Np - (d.sb & (d.Np - 1)) + (d.Np >> 1)) & (d.Np - 1);
    const int32_t o = (int32_t)dd - (int32_t)(d.Np >> 1);
    const uint32_t i = index_at(d, j, o);
#pragma unroll
    for (int l = 0; l < kMaxHash - 1; ++l)
        if ((uint32_t)l < L && fabsf(hypotf(u[l + 1].x, u[l + 1].y) - mag0) > d.iso_tol_f * mag0) return 0;
    if (Ents::kDirect) {
        *oi = (uint32_t)o;
        return 1;
    }
    const uint32_t oa = (uint32_t)(o < 0 ? -o : o);
    const double gain = d.wtab[oa];
    const double gi = d.winv ? d.winv[oa] : 0.0;  // loaded beside the gain: one memory latency for both
    if (!(gain >= d.gmin)) return 0;
    *oi = i;
    *gout = gain;
    *ginv = gi;
    return 1;
}

// The FP64 data path's decisions, taken in FP32 wherever FP64 must agree.  The rounding of a subtracted
// bin to FP32, hypotf and atan2f move a magnitude by less than 3e-7 of itself and a phase by less than
// 2.5e-7 of a turn; a comparison or rounding that lies within several times that of its boundary (kMagGuard,
// kPhaseGuard32) is not taken and the whole bin goes through decode_bin_fp64.  Every other one has the same
// outcome in both, so the decode is that of decode_bin_fp64 (about 200 FP64 operations per bin and warp at
// 1/64 of the FP32 rate).  Values stay in FP64.
constexpr float kMagGuard = 2e-6f, kPhaseGuard32 = 1e-6f;
// -1: m < t, 1: m > t, 0: too close (also among the denormal numbers, whose rounding is not relative)
__device__ __forceinline__ int cmp_guarded(float m, float t) {
    const float g = fmaf(kMagGuard, t, 1e-36f);
    return m > t + g ? 1 : (m < t - g ? -1 : 0);
}
constexpr int kUndecided = -1;
template <typename Ents>
__device__ __forceinline__ int decode_bin_guarded(const DecodeCtx& d, uint32_t j, const double2* u, const Ents& ents,
                                                  uint32_t* oi, double* gout, double* ginv, bool* above) {
    float2 v[kMaxHash];
    const uint32_t L = d.H - 1;
#pragma unroll
    for (int h = 0; h < kMaxHash; ++h)
        v[h] = (uint32_t)h < d.H ? make_float2((float)u[h].x, (float)u[h].y) : make_float2(0.f, 0.f);
    *ginv = 0.0;
    *above = false;
    const float mag0 = hypotf(v[0].x, v[0].y);
    // thresholds and magnitudes that FP32 holds to full precision only
    if (!(d.thr_f > 1e-15f && d.thr_f < 1e15f && mag0 < 1e18f)) return kUndecided;
    const int over = cmp_guarded(mag0, d.thr_f);
    if (over == 0) return kUndecided;
    if (over < 0) {
        if (!ents.any()) return 0;
        const int lo = cmp_guarded(mag0, d.ref_lo_f), hi = cmp_guarded(mag0, d.ref_hi_f);
        return lo < 0 || hi > 0 ? 0 : kUndecided;  // (a re-estimation is decided in FP64)
    }
    *above = true;
    float ml[kMaxHash - 1], th[kMaxHash - 1];
#pragma unroll
    for (int l = 0; l < kMaxHash - 1; ++l)
        if ((uint32_t)l < L) {
            ml[l] = hypotf(v[l + 1].x, v[l + 1].y);
            th[l] = phase01_f(mul_conj_f(v[0], v[l + 1]));
        }
    // a hashing far below u_0 passes a wide isolation tolerance only; FP32 may not hold its product's phase
    if (d.iso_tol_f > 0.5f) {
#pragma unroll
        for (int l = 0; l < kMaxHash - 1; ++l)
            if ((uint32_t)l < L && !(ml[l] > 1e-30f && ml[l] * mag0 > 1e-30f)) return kUndecided;
    }
    // location ladder, coarsest shift first: each rounding has to stay clear of a half
    uint32_t c = 0, logM = 0;
#pragma unroll
    for (int l = kMaxHash - 2; l >= 0; --l) {
        if ((uint32_t)l >= L) continue;
        const uint32_t logMp = d.logNp - d.logR[l], logRatio = logMp - logM;  // from logM = 0: the coarsest, c = 0
        const float y = th[l] * pow2_f((int)logRatio) - __uint2float_rn(c) * pow2_f(-(int)logM);
        const float f = y - floorf(y);
        if (!(fabsf(f - 0.5f) > kPhaseGuard32 * (pow2_f((int)logRatio) + 1.0f))) return kUndecided;
        c += ((uint32_t)__float2int_rd(y + 0.5f) & ((1u << logRatio) - 1u)) << logM;
        logM = logMp;
    }
    const uint32_t dd = (c + d.Np - (d.sb & (d.Np - 1)) + (d.Np >> 1)) & (d.Np - 1);
    const int32_t o = (int32_t)dd - (int32_t)(d.Np >> 1);
#pragma unroll
    for (int l = 0; l < kMaxHash - 1; ++l)
        if ((uint32_t)l < L) {
            const float df = fabsf(ml[l] - mag0), t = d.iso_tol_f * mag0, g = kMagGuard * (mag0 + ml[l]);
            if (df > t + g) return 0;
            if (!(df < t - g)) return kUndecided;
        }
    if (Ents::kDirect) {
        *oi = (uint32_t)o;
        return 1;
    }
    const double gain = d.wtab[o < 0 ? -o : o];
    if (!(gain >= d.gmin)) return 0;
    *oi = index_at(d, j, o);
    *gout = gain;
    return 1;
}

template <typename Ents>
__device__ __forceinline__ int decode_bin(const DecodeCtx& d, uint32_t j, const double2* u, const Ents& ents,
                                          const uint32_t* ent_idx, const double* ent_gain, uint32_t* oi,
                                          double* gout, double* ginv, bool* above) {
    const int kind = decode_bin_guarded(d, j, u, ents, oi, gout, ginv, above);
    return kind != kUndecided ? kind : decode_bin_fp64(d, j, u, ents, ent_idx, ent_gain, oi, gout, ginv, above);
}
template <typename Ents>
__device__ __forceinline__ int decode_bin(const DecodeCtx& d, uint32_t j, const float2* u, const Ents& ents,
                                          const uint32_t* ent_idx, const double* ent_gain, uint32_t* oi,
                                          double* gout, double* ginv, bool* above) {
    return decode_bin_fp32(d, j, u, ents, ent_idx, ent_gain, oi, gout, ginv, above);
}

__device__ __forceinline__ MaskEntries bin_entries(std::true_type, const uint32_t* words, uint32_t stride, uint32_t nwords,
                                                   const uint32_t*, const uint32_t*) {
    return MaskEntries{words, stride, nwords};
}
__device__ __forceinline__ ListEntries bin_entries(std::false_type, const uint32_t*, uint32_t, uint32_t, const uint32_t* list,
                                                   const uint32_t* start) {
    return ListEntries{list + start[0], start[1] - start[0]};
}

// Bin j's hashings after the subtraction of zhat, for the decisions: u_h = U_h - sum over the bin's
// entries e (in list order) of sub[e H + h], in the data path's precision (FP64 terms and sums for
// the FP64 path; the terms rounded to FP32 and summed in FP32 for the FP32 path, whose bins carry
// ~1e-6 of rounding).  The values of decoded bins are formed separately from subtracted_u0 in FP64.
template <typename Ents>
__device__ __forceinline__ void subtracted_bin(const double2* U, uint32_t B, uint32_t H, uint32_t j, const Ents& ents,
                                               const double2* sub, const float2* /*sub_f*/, double2* u) {
    for (uint32_t h = 0; h < H; ++h) {
        double2 w = U[h * B + j];
        ents.each([&](uint32_t e) {
            w.x -= sub[e * H + h].x;
            w.y -= sub[e * H + h].y;
        });
        u[h] = w;
    }
}
template <typename Ents>
__device__ __forceinline__ void subtracted_bin(const float2* U, uint32_t B, uint32_t H, uint32_t j, const Ents& ents,
                                               const double2* /*sub*/, const float2* sub_f, float2* u) {
#pragma unroll
    for (int h = 0; h < kMaxHash; ++h) u[h] = (uint32_t)h < H ? U[h * B + j] : make_float2(0.0f, 0.0f);
    ents.each([&](uint32_t e) {
        const float2* t = sub_f + e * H;
#pragma unroll
        for (int h = 0; h < kMaxHash; ++h)
            if ((uint32_t)h < H) {
                u[h].x -= t[h].x;
                u[h].y -= t[h].y;
            }
    });
}
// u_0 of bin j after the subtraction, in FP64 (the first row of subtracted_bin, same order); entry e's
// FP64 term of hashing 0 is sub[e * stride]
template <typename C, typename Ents>
__device__ __forceinline__ double2 subtracted_u0(const C* U, uint32_t stride, uint32_t j, const Ents& ents,
                                                 const double2* sub) {
    const C v = U[j];
    double2 w = make_double2((double)v.x, (double)v.y);
    ents.each([&](uint32_t e) {
        w.x -= sub[e * stride].x;
        w.y -= sub[e * stride].y;
    });
    return w;
}

// ------------------------------------------------------------------------------------------------
// The round kernel
// ------------------------------------------------------------------------------------------------
template <typename R>
__device__ void gather_fold(const ExactArgs& a, const void* xrow, uint32_t xmask, uint32_t s, uint32_t c,
                            uint32_t sigma, uint32_t b, unsigned char* smem) {
    using C = typename Cx<R>::T;
    C* stage = reinterpret_cast<C*>(smem);
    C* red = stage + a.stage;
    const uint32_t tid = threadIdx.x;
    const C* __restrict__ x = reinterpret_cast<const C*>(xrow);
    const R* __restrict__ taps = taps_of<R>(a);
    const int64_t t_lo = -a.T + (int64_t)c * a.ctaps;
    const int64_t t_hi = min(t_lo + (int64_t)a.ctaps, a.T + 1);
    const uint32_t ntap = (uint32_t)(t_hi - t_lo);
    const int32_t base = (int32_t)(t_lo - (int64_t)a.a_base - (int64_t)a.maxshift);  // sample held by stage[0]
    const uint32_t cnt = ntap + a.maxshift;
    // step 1a: gather the sigma-strided samples x_{sigma s}, s in [base, base + cnt) (12 loads in flight)
#ifndef SFFT_GATHER_IN_FLIGHT
#define SFFT_GATHER_IN_FLIGHT 12
#endif
    constexpr int kInFlight = SFFT_GATHER_IN_FLIGHT;
    for (uint32_t i0 = tid; i0 < cnt; i0 += kThreads * kInFlight) {
        C v[kInFlight];
#pragma unroll
        for (int q = 0; q < kInFlight; ++q) {
            const uint32_t i = i0 + (uint32_t)q * kThreads;
            if (i < cnt) v[q] = ldg_c(x + ((sigma * (uint32_t)(base + (int32_t)i)) & xmask));
        }
#pragma unroll
        for (int q = 0; q < kInFlight; ++q) {
            const uint32_t i = i0 + (uint32_t)q * kThreads;
            if (i < cnt) stage[i] = v[q];
        }
    }
    const bool big = a.B > (uint32_t)kThreads;
    if (big)
        for (uint32_t i = tid; i < a.H * a.B; i += kThreads) red[i] = mkc((R)0, (R)0);
    __syncthreads();
    // step 1b + 2: y_t = G_t x_{sigma (t - a_h)} w^{sigma b t}, folded mod B
    C acc[kMaxHash];
#pragma unroll
    for (int h = 0; h < kMaxHash; ++h) acc[h] = mkc((R)0, (R)0);
    const uint32_t sb = sigma * b;
    const R inv_half_n = (R)2 / (R)a.n;
    for (uint32_t k = tid; k < ntap; k += kThreads) {
        const int32_t t = (int32_t)t_lo + (int32_t)k;
        const R g = taps[t < 0 ? -t : t];
        const C gt = tap_factor(a, g, sb * (uint32_t)t, inv_half_n);
        const uint32_t si = k + a.maxshift;
        if (!big) {
#pragma unroll
            for (int h = 0; h < kMaxHash; ++h)
                if ((uint32_t)h < a.H) acc[h] = cfma(gt, stage[si - a.a[h]], acc[h]);
        } else {
            const uint32_t r = (uint32_t)t & (a.B - 1);
            for (uint32_t h = 0; h < a.H; ++h) red[h * a.B + r] = cfma(gt, stage[si - a.a[h]], red[h * a.B + r]);
        }
    }
    if (!big) {
        for (uint32_t h = 0; h < a.H; ++h) red[h * kThreads + tid] = acc[h];
    }
    __syncthreads();
    C* part = reinterpret_cast<C*>(a.part) + (size_t)s * a.part_stride + (size_t)c * a.H * a.B;
    if (!big) {
        // residue of thread tid is (t_lo + tid) mod B; the threads of residue r are owner + m B
        for (uint32_t r = tid; r < a.B; r += kThreads) {
            const uint32_t owner = (r - (uint32_t)t_lo) & (a.B - 1);
            for (uint32_t h = 0; h < a.H; ++h) {
                C sum = mkc((R)0, (R)0);
                for (uint32_t m = owner; m < (uint32_t)kThreads; m += a.B) sum = cadd(sum, red[h * kThreads + m]);
                part[h * a.B + r] = sum;
            }
        }
    } else {
        for (uint32_t i = tid; i < a.H * a.B; i += kThreads) part[i] = red[i];
    }
}

// The same fold with a CTA owning kOwnerRes residues of the round (rounds of kThreads bins or more of
// large plans), so that no partial fold leaves the CTA (B = 4096 has about 140 chunks, whose partial folds
// one CTA would have to add).  Four threads load a residue's taps, a batch of loads ahead of the fold; the
// taps' factors are formed once into shared memory, and thread (residue, h) folds hashing h.  The ladder's
// shifts are multiples of B, so the samples of every hashing's tap t, x_{sigma (t - a_h)}, are the
// residue's own: the last ones stay in its column of the ring.  Order of the sums: that of the chunks (a
// residue's taps of a chunk from zero, then the chunks in order), so the bits are the same.
// Bound by random sectors.  64 residues a CTA, not 256: at n = 2^22, k = 227, batch 33 round 0 then has
// more CTAs than the chip has places and ends before the later rounds' gathers share the bandwidth.
template <typename R>
__device__ __forceinline__ void gather_owner(const ExactArgs& a, const void* xrow, uint32_t xmask, uint32_t s,
                                             uint32_t blk, uint32_t sigma, uint32_t b, unsigned char* smem) {
    using C = typename Cx<R>::T;
    constexpr uint32_t kLoads = owner_loads<R>(), kQ = kThreads / kOwnerRes, kBatch = kLoads * kQ;
    const uint32_t lr = threadIdx.x & (kOwnerRes - 1), q = threadIdx.x / kOwnerRes, B = a.B, H = a.H;
    C* ring = reinterpret_cast<C*>(smem) + lr;      // [a.ring][kOwnerRes], this residue's column
    C* factor = ring + (size_t)a.ring * kOwnerRes;  // [kBatch][kOwnerRes]
    const uint32_t rmask = a.ring - 1u;
    const C* __restrict__ x = reinterpret_cast<const C*>(xrow);
    const R* __restrict__ taps = taps_of<R>(a);
    const uint32_t first = blk * kOwnerRes, i0 = first + lr;  // first tap -T + i0, then every B-th
    const uint32_t ntot = (uint32_t)(2 * a.T + 1);
    const uint32_t mend = first < ntot ? (ntot - first + B - 1) / B : 0;  // taps per residue, rounded up for all
    const uint32_t mine = i0 < ntot ? (ntot - i0 + B - 1) / B : 0;        // this one's
    const uint32_t nt = a.ctaps > B ? a.ctaps / B : 1u;       // a residue's taps per chunk
    const uint32_t t0 = (uint32_t)(int32_t)(-a.T) + i0;
    const uint32_t dmax = a.maxshift / B;                     // sample j of the residue: t0 + (j - dmax) B
    const uint32_t dl = dmax - (q < H ? a.a[q] / B : 0u);     // hashing q's tap m takes sample m + dl
    const uint32_t x0 = sigma * (t0 - a.maxshift), xstep = sigma * B, sb = sigma * b;
    const R inv_half_n = (R)2 / (R)a.n;
    C acc = mkc((R)0, (R)0), sum = acc;
    for (uint32_t j = q; j < dmax; j += kQ) ring[(j & rmask) * kOwnerRes] = ldg_c(x + ((x0 + j * xstep) & xmask));
    C v[kLoads];
    R g[kLoads];
    auto load = [&](uint32_t m0) {
#pragma unroll
        for (uint32_t u = 0; u < kLoads; ++u) {
            const uint32_t m = m0 + q + u * kQ;
            if (m < mine) {
                v[u] = ldg_c(x + ((x0 + (m + dmax) * xstep) & xmask));
                const int32_t t = (int32_t)(t0 + m * B);
                g[u] = taps[t < 0 ? -t : t];
            }
        }
    };
    load(0);
    for (uint32_t m0 = 0; m0 < mend; m0 += kBatch) {
#pragma unroll
        for (uint32_t u = 0; u < kLoads; ++u) {
            const uint32_t m = m0 + q + u * kQ;
            if (m < mine) {
                ring[((m + dmax) & rmask) * kOwnerRes] = v[u];
                factor[(m - m0) * kOwnerRes] = tap_factor(a, g[u], sb * (t0 + m * B), inv_half_n);
            }
        }
        __syncthreads();
        if (m0 + kBatch < mend) load(m0 + kBatch);
        if (q < H) {
            const uint32_t mb = min(m0 + kBatch, mine);
            // (a short loop: unrolled, its code is fetched from L2 by every SM for as long as it runs)
#pragma unroll 2
            for (uint32_t m = m0; m < mb; ++m) {
                if (m != 0 && (m & (nt - 1)) == 0) {
                    sum = cadd(sum, acc);
                    acc = mkc((R)0, (R)0);
                }
                acc = cfma(factor[(m - m0) * kOwnerRes], ring[((m + dl) & rmask) * kOwnerRes], acc);
            }
        }
        __syncthreads();  // the ring and the factors are written again
    }
    if (q < H) {  // bit-reversed, as the bin FFT takes it
        C* area = reinterpret_cast<C*>(a.part) + (size_t)s * a.part_stride + (__brev(t0 & (B - 1)) >> (32u - a.logB));
        area[(size_t)q * B] = cadd(sum, acc);
    }
}

// |v| < prune thr in FP64, by FP32 where that is clear of the bound
__device__ __forceinline__ bool dropped(double2 v, const ExactArgs& a) {
    const float f = hypotf((float)v.x, (float)v.y);
    if (a.drop_f > 1e-25f && a.drop_f < 1e25f && f < 1e18f) {
        const int c = cmp_guarded(f, a.drop_f);
        if (c != 0) return c < 0;
    }
    return cmag(v) < a.prune * a.thr;
}

// Step 2 across chunks: U[h][brev(r)] = sum over chunks c, in order, of part[c][h][r].  Each thread
// takes E elements of up to CM chunks with all their loads in flight at once (CM >= chunks), else
// one element at a time in batches of 16.
template <int E, int CM, typename C>
__device__ __forceinline__ void sum_partials_batched(const C* part, uint32_t chunks, uint32_t H, uint32_t logB, C* U) {
    const uint32_t B = 1u << logB, HB = H * B, shift_br = 32u - logB;
    for (uint32_t i0 = threadIdx.x; i0 < HB; i0 += (uint32_t)kThreads * E) {
        C v[E][CM];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = i0 + (uint32_t)e * kThreads;
            const uint32_t h = i >> logB, r = i & (B - 1);
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (i < HB && (uint32_t)c < chunks) v[e][c] = __ldcg(part + ((size_t)c * H + h) * B + r);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t i = i0 + (uint32_t)e * kThreads;
            if (i < HB) {
                C sum;
                sum.x = 0;
                sum.y = 0;
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if ((uint32_t)c < chunks) sum = cadd(sum, v[e][c]);
                U[(i >> logB) * B + (__brev(i & (B - 1)) >> shift_br)] = sum;
            }
        }
    }
}
template <typename C>
__device__ void sum_partials(const C* part, uint32_t chunks, uint32_t H, uint32_t logB, C* U) {
    constexpr bool f32 = sizeof(C) == sizeof(float2);  // FP64 bins: half the loads in flight (registers)
    if (chunks <= 8) {
        sum_partials_batched<f32 ? 2 : 1, 8>(part, chunks, H, logB, U);
    } else if (chunks <= 16) {
        sum_partials_batched<1, 16>(part, chunks, H, logB, U);
    } else {
        const uint32_t B = 1u << logB, shift_br = 32u - logB;
        for (uint32_t i = threadIdx.x; i < H * B; i += kThreads) {
            const uint32_t h = i >> logB, r = i & (B - 1);
            C sum;
            sum.x = 0;
            sum.y = 0;
            for (uint32_t c0 = 0; c0 < chunks; c0 += 16) {  // 16 loads in flight, summed in chunk order
                C v[16];
#pragma unroll
                for (uint32_t q = 0; q < 16; ++q)
                    if (c0 + q < chunks) v[q] = __ldcg(part + ((size_t)(c0 + q) * H + h) * B + r);
#pragma unroll
                for (uint32_t q = 0; q < 16; ++q)
                    if (c0 + q < chunks) sum = cadd(sum, v[q]);
            }
            U[h * B + (__brev(r) >> shift_br)] = sum;
        }
    }
}

// Parts of a round's finisher: the bins (partial folds summed in chunk order, bit-reversed, B-point
// FFT) and the decode (zhat subtraction, location, estimation, merge).  kFinBins leaves the bins in
// the first H B entries of the request's partial-fold area of the round; kFinDecode starts from there.
enum FinPart { kFinBins = 1, kFinDecode = 2, kFinAll = 3 };

template <bool LARGE>
__device__ __forceinline__ void fft_rows(const ExactArgs& a, float2* U) {
    if (LARGE)
        fft_rows_by_passes(U, a.H, a.logB);
    else
        block_fft_rows<float>(U, a.H, a.logB);
}
template <bool LARGE>
__device__ __forceinline__ void fft_rows(const ExactArgs& a, double2* U) {
    fft_rows_fp64(U, a.H, a.logB, a.logn, a.tw, a.tw_shift);
}

// KIND (see DecodeKind): how the entries of a bin are found; kDecodeLarge only forms the bins here
template <typename R, int KIND = kDecodeLists>
__device__ bool finish_round(const ExactArgs& a, uint32_t s, uint32_t sigma, uint32_t b, unsigned char* smem,
                             int part = kFinAll, bool carry = false, bool bins_here = false,
                             const uint32_t* next_ctr = nullptr) {
    using C = typename Cx<R>::T;
    const uint32_t tid = threadIdx.x;
    const uint32_t B = a.B, H = a.H;
    constexpr bool masks = KIND == kDecodeMasks;
    const FinLayout Ly = fin_layout(B, H, a.zcap, sizeof(C), masks);
    C* U = reinterpret_cast<C*>(smem + Ly.U);
    uint32_t* ent_idx = reinterpret_cast<uint32_t*>(smem + Ly.ent_idx);
    uint32_t* ent_bin = reinterpret_cast<uint32_t*>(smem + Ly.ent_bin);
    double2* ent_val = reinterpret_cast<double2*>(smem + Ly.ent_val);
    double* ent_gain = reinterpret_cast<double*>(smem + Ly.ent_gain);
    double2* ent_sub = reinterpret_cast<double2*>(smem + Ly.ent_sub);
    float2* ent_sub_f = reinterpret_cast<float2*>(smem + Ly.ent_sub_f);
    uint32_t* mask = reinterpret_cast<uint32_t*>(smem + Ly.mask);  // [word][B]: bit e mod 32 of word e / 32
    uint32_t* bin_cnt = reinterpret_cast<uint32_t*>(smem + Ly.bin_cnt);
    uint32_t* bin_start = reinterpret_cast<uint32_t*>(smem + Ly.bin_start);
    uint32_t* bin_list = reinterpret_cast<uint32_t*>(smem + Ly.bin_list);
    uint32_t* cand_idx = reinterpret_cast<uint32_t*>(smem + Ly.cand_idx);
    double2* cand_val = reinterpret_cast<double2*>(smem + Ly.cand_val);
    uint32_t* srt_idx = reinterpret_cast<uint32_t*>(smem + Ly.srt_idx);
    double2* srt_val = reinterpret_cast<double2*>(smem + Ly.srt_val);
    uint32_t* out_idx = reinterpret_cast<uint32_t*>(smem + Ly.out_idx);
    double2* out_val = reinterpret_cast<double2*>(smem + Ly.out_val);
    uint32_t* keep = reinterpret_cast<uint32_t*>(smem + Ly.keep);
    uint32_t* scan = reinterpret_cast<uint32_t*>(smem + Ly.scan);
    __shared__ uint32_t s_nw, s_above, s_kept;
    C* area = reinterpret_cast<C*>(a.part) + (size_t)s * a.part_stride;  // the round's partial folds

    // steps 2 (across chunks) and 3: partial folds summed in chunk order, bit-reversed, FFT
    if (part & kFinBins) {
        if (KIND == kDecodeLarge && a.owner)
            load_rows(U, area, H * B);  // whole folds, bit-reversed
        else
            sum_partials(area, a.chunks, H, a.logB, U);
        fft_rows<KIND == kDecodeLarge>(a, U);  // starts and ends with a barrier
        if (!(part & kFinDecode)) {  // every partial fold has been read: the area takes the bins
            for (uint32_t i = tid; i < H * B; i += kThreads) area[i] = U[i];
            return false;
        }
    }
    // The round's bins, when another CTA formed them (bins_here: this CTA did, just before, in place),
    // read through L2 only: each thread's first four are loaded here and stored after the entries'
    // window gains below have been requested, so that both wait out one memory latency.  The last
    // thread reads the next round's second counter (next_ctr) with an acquire load alongside: if that
    // round's bins have arrived, the caller goes on to its decode without an arrival (next_ready).
    __shared__ uint32_t s_next_ready;
    const bool load_U = !(part & kFinBins) && !bins_here;
    C uv[4];
    if (load_U) {
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (tid + q * kThreads < H * B) uv[q] = __ldcg(area + tid + q * kThreads);
    }
    if (tid == kThreads - 1 && next_ctr != nullptr) s_next_ready = acquire_is(next_ctr, 1u) ? 1u : 0u;

    if (masks) {
        for (uint32_t i = tid; i < B * ((a.zcap + 31) / 32); i += kThreads) mask[i] = 0;
        __syncthreads();  // (waits for nothing: the loads above are still on their way)
    }
    // zhat of this request and its per-entry subtraction terms
    // zhat is read through L2 only: in the one-launch path another CTA of this launch wrote it
    // (the first entry of each thread is fetched together with the count)
    // zhat of the previous round stays in this CTA's shared memory (up to kCarry entries) when the
    // previous round's decode of this request ran here (carry): no global load for it then
    __shared__ uint32_t c_idx[kCarry];
    __shared__ double2 c_val[kCarry];
    __shared__ uint32_t c_n;
    const bool use_carry = carry && !a.bins_only && a.zcap <= kCarry;
    const uint32_t zlim = a.bins_only ? a.e_nz : a.zcap;
    uint32_t zi0 = 0;
    double2 zv0 = make_double2(0.0, 0.0);
    if (use_carry) {
        if (tid < c_n) {
            zi0 = c_idx[tid];
            zv0 = c_val[tid];
        }
    } else if (tid < zlim) {
        zi0 = __ldcg(a.zidx + (size_t)s * a.zcap + tid);
        zv0 = __ldcg(a.zval + (size_t)s * a.zcap + tid);
    }
    const uint32_t nz = a.bins_only ? a.e_nz : (use_carry ? c_n : min(__ldcg(a.zcount + s), a.zcap));
    // the decode context is the same for every thread: one copy in shared memory (registers would
    // hold it only by spilling it to local memory)
    __shared__ DecodeCtx d;
    if (tid == kThreads - 2) fill_ctx_round(d, a, sigma, b);
    // (the entries need no part of d: their window gains are read while it is filled, by a thread that
    // holds no entry unless zhat has more than kThreads - 2)
    const uint32_t Np = (uint32_t)(a.n >> a.logB), logNp = ilog2_u32(Np);
    // The FP32 data path keeps FP64 work (issued at a small fraction of the FP32 rate) to the values:
    // entry e's FP64 term of hashing 0 goes to ent_sub[e] and its gain-scaled value, rounded to FP32,
    // to ent_gz[e] (behind the first zcap entries of ent_sub; H >= 2 outside single-hashing mode); the
    // terms of the decisions are formed in FP32 from there.  The FP64 path forms every term in FP64.
    constexpr bool f32 = sizeof(C) == sizeof(float2);
    float2* ent_gz = reinterpret_cast<float2*>(ent_sub + a.zcap);
    const uint32_t a0 = a.a_base + a.a[0];
    for (uint32_t e = tid; e < nz; e += kThreads) {
        const uint32_t i = e == tid ? zi0 : (use_carry ? c_idx[e] : __ldcg(a.zidx + (size_t)s * a.zcap + e));
        const double2 v = e == tid ? zv0 : (use_carry ? c_val[e] : __ldcg(a.zval + (size_t)s * a.zcap + e));
        ent_idx[e] = i;
        ent_val[e] = v;
        uint32_t jb;
        const int32_t o = offset_of((sigma * (i - b)) & a.nmask, Np, logNp, a.nmask, &jb);
        if (masks)
            atomicOr(&mask[(e >> 5) * B + jb], 1u << (e & 31u));
        else
            ent_bin[e] = jb;
        const double gain = a.wtab[o < 0 ? -o : o];
        ent_gain[e] = gain;
        if (f32) {
            const double2 gz = make_double2(gain * v.x, gain * v.y);
            double2 t0 = gz;  // hashing 0 has offset 0 in the transform's rounds: w^0 = 1
            const uint32_t e0 = (a0 * sigma * i) & a.nmask;
            if (e0 != 0) {
                const double2 w = term_root<R>(a, e0);
                t0 = make_double2(gz.x * w.x - gz.y * w.y, gz.x * w.y + gz.y * w.x);
            }
            ent_sub[e] = t0;
            if (!a.bins_only) ent_gz[e] = make_float2((float)gz.x, (float)gz.y);
        }
    }
    if (load_U) {
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (tid + q * kThreads < H * B) U[tid + q * kThreads] = uv[q];
        for (uint32_t i0 = tid + 4 * kThreads; i0 < H * B; i0 += 4 * kThreads) {  // B > kThreads
            C v[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q)
                if (i0 + q * kThreads < H * B) v[q] = __ldcg(area + i0 + q * kThreads);
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q)
                if (i0 + q * kThreads < H * B) U[i0 + q * kThreads] = v[q];
        }
    }
    if (tid == 0) {
        s_nw = 0;
        s_above = 0;
        s_kept = 0;
    }
    __syncthreads();  // d, the entries and the counts
    // read here, before thread 0 can reach the next round's write
    const bool next_ready = next_ctr != nullptr && s_next_ready != 0;
    // step 4 terms: W(-o(i)) zhat_i w^{a_h sigma i} for every (entry, hashing)
    if (f32) {
        if (!a.bins_only) {
            const float two_over_n = 2.0f * d.inv_n_f;  // exact: n is a power of two
            for (uint32_t q = tid; q < nz * H; q += kThreads) {
                const uint32_t e = q / H, h = q - e * H;
                const uint32_t ex = ((a.a_base + a.a[h]) * sigma * ent_idx[e]) & a.nmask;
                const int32_t es = ex > (a.nmask >> 1) ? (int32_t)((int64_t)ex - (int64_t)a.n) : (int32_t)ex;
                float sn, cs;
                sincospif((float)es * two_over_n, &sn, &cs);
                const float2 g = ent_gz[e];  // times w = (cs, -sn)
                ent_sub_f[q] = make_float2(g.x * cs + g.y * sn, g.y * cs - g.x * sn);
            }
        }
    } else {
        for (uint32_t q = tid; q < nz * H; q += kThreads) {
            const uint32_t e = q / H, h = q - e * H;
            const uint32_t i = ent_idx[e];
            const double2 w = term_root<R>(a, ((a.a_base + a.a[h]) * sigma * i) & a.nmask);
            const double2 gz = make_double2(ent_gain[e] * ent_val[e].x, ent_gain[e] * ent_val[e].y);
            ent_sub[q] = make_double2(gz.x * w.x - gz.y * w.y, gz.x * w.y + gz.y * w.x);
        }
    }
    const uint32_t sub_stride = f32 ? 1u : H;  // where subtracted_u0 finds hashing 0's FP64 terms
    if (masks)
        __syncthreads();  // the terms
    else
        bucket_entries(ent_bin, nz, B, bin_cnt, bin_start, bin_list, scan);  // (a barrier before the terms are read)
    if (a.bins_only) {  // single-hashing mode: the subtracted bins u_0 in FP64, no decode
        for (uint32_t j = tid; j < B; j += kThreads)
            a.ubins[j] =
                subtracted_u0(U, sub_stride, j, ListEntries{bin_list + bin_start[j], bin_start[j + 1] - bin_start[j]},
                              ent_sub);
        return false;
    }
    // step 4 and the decode, one bin per thread: decisions in the data path's precision
    for (uint32_t j = tid; j < B; j += kThreads) {
        C u[kMaxHash];
        const auto ents = bin_entries(std::integral_constant<bool, masks>(), mask + j, B, (nz + 31) / 32, bin_list, bin_start + j);
        subtracted_bin(U, B, H, j, ents, ent_sub, ent_sub_f, u);
        uint32_t oi = 0;
        double gain = 1.0, ginv = 0.0;
        bool above;
        const int kind = decode_bin(d, j, u, ents, ent_idx, ent_gain, &oi, &gain, &ginv, &above);
        // counts and candidate slots, one shared-memory atomic per warp and counter
        const unsigned m = __activemask();
        const unsigned ma = __ballot_sync(m, above), mk = __ballot_sync(m, kind == 1), mw = __ballot_sync(m, kind != 0);
        const uint32_t lane = tid & 31u, leader = (uint32_t)__ffs((int)m) - 1u;
        uint32_t base = 0;
        if (lane == leader) {
            if (ma) atomicAdd(&s_above, (uint32_t)__popc((int)ma));
            if (mk) atomicAdd(&s_kept, (uint32_t)__popc((int)mk));
            if (mw) base = atomicAdd(&s_nw, (uint32_t)__popc((int)mw));
        }
        base = __shfl_sync(m, base, (int)leader);
        if (kind != 0) {
            const uint32_t slot = base + (uint32_t)__popc((int)(mw & ((1u << lane) - 1u)));
            cand_idx[slot] = oi;
            // its value: u_0 (step 4 in FP64) / W(-o), as a product with 1 / W(-o) from the table where
            // the decode read one (FP32 path), else as a quotient
            const double2 u0 = subtracted_u0(U, sub_stride, j, ents, ent_sub);
            if (f32 && kind == 1 && d.winv)
                cand_val[slot] = make_double2(u0.x * ginv, u0.y * ginv);
            else
                cand_val[slot] = make_double2(u0.x / gain, u0.y / gain);
        }
    }
    __syncthreads();
    const uint32_t nw = s_nw;

    const bool last = a.last_round != 0;
    if (nw == 0) {
        // nothing decoded: zhat stays as it is (its entries passed the same prune test when merged)
        if (!a.bins_only && a.zcap <= kCarry && !use_carry) {  // this CTA keeps it for the next round
            for (uint32_t e = tid; e < nz; e += kThreads) {
                c_idx[e] = ent_idx[e];
                c_val[e] = ent_val[e];
            }
            if (tid == 0) c_n = nz;
        }
        if (last) {
            for (uint32_t e = tid; e < nz && e < a.out_cap; e += kThreads) {
                a.out_idx[(size_t)s * a.out_cap + e] = ent_idx[e];
                a.out_val[(size_t)s * a.out_cap + e] = ent_val[e];
            }
            if (tid == 0) {
                a.out_count[s] = nz < a.out_cap ? nz : a.out_cap;
                int32_t flag = SFFT_OK;
                if (__ldcg(a.zflag + s) || nz > a.out_cap)
                    flag = SFFT_ERR_CAPACITY;
                else if (s_above > s_kept)
                    flag = SFFT_ERR_NOT_CONVERGED;
                a.out_flag[s] = flag;
            }
        }
        return next_ready;
    }
    // merge what into zhat (NoiselessSparseFFT: zhat <- zhat + what), zhat first on equal indices,
    // then drop entries below prune * thr
    const uint32_t tot = nz + nw;
    if (nw <= (uint32_t)kThreads) {
        // positions by counting (the candidates' indices are distinct): zhat entry e goes to e + the
        // number of candidates below its index, candidate c to the number of candidates below its
        // index + the number of zhat entries at or below it
        for (uint32_t e = tid; e < nz; e += kThreads) {
            const uint32_t key = ent_idx[e];
            uint32_t r = 0;
            for (uint32_t q = 0; q < nw; ++q) r += cand_idx[q] < key ? 1u : 0u;
            out_idx[e + r] = key;
            out_val[e + r] = ent_val[e];
        }
        if (tid < nw) {
            const uint32_t key = cand_idx[tid];
            uint32_t r = 0;
            for (uint32_t q = 0; q < nw; ++q) r += cand_idx[q] < key ? 1u : 0u;
            const uint32_t pos = r + upper_bound_u32(ent_idx, nz, key);
            out_idx[pos] = key;
            out_val[pos] = cand_val[tid];
        }
    } else {  // many candidates: sorted first, then placed by binary searches
        rank_sort(cand_idx, cand_val, nw, srt_idx, srt_val);
        for (uint32_t e = tid; e < nz; e += kThreads) {
            const uint32_t pos = e + lower_bound_u32(srt_idx, nw, ent_idx[e]);
            out_idx[pos] = ent_idx[e];
            out_val[pos] = ent_val[e];
        }
        for (uint32_t c = tid; c < nw; c += kThreads) {
            const uint32_t pos = c + upper_bound_u32(ent_idx, nz, srt_idx[c]);
            out_idx[pos] = srt_idx[c];
            out_val[pos] = srt_val[c];
        }
    }
    __syncthreads();
    // a merged entry's fate: heads of equal indices take their duplicate's value, small ones are dropped
    auto keep_merged = [&](uint32_t p, uint32_t idx, double2& v) -> bool {
        if (p != 0 && out_idx[p - 1] == idx) return false;
        if (p + 1 < tot && out_idx[p + 1] == idx) {
            v.x += out_val[p + 1].x;
            v.y += out_val[p + 1].y;
        }
        // |v| < prune thr, in the data path's precision (FP32: against prune thr rounded up)
        return f32 ? !(hypotf((float)v.x, (float)v.y) < a.drop_f) : !dropped(v, a);
    };
    uint32_t* zi = a.zidx + (size_t)s * a.zcap;
    double2* zv = a.zval + (size_t)s * a.zcap;
    auto put = [&](uint32_t pos, uint32_t idx, double2 v) {
        if (pos < a.zcap) {
            zi[pos] = idx;
            zv[pos] = v;
            if (a.zcap <= kCarry) {
                c_idx[pos] = idx;
                c_val[pos] = v;
            }
        }
        if (last && pos < a.out_cap) {
            a.out_idx[(size_t)s * a.out_cap + pos] = idx;
            a.out_val[(size_t)s * a.out_cap + pos] = v;
        }
    };
    uint32_t newcount = 0;
    if (tot <= (uint32_t)kThreads) {  // one merged entry per thread: a ballot and one barrier
        uint32_t idx = 0;
        double2 v = make_double2(0.0, 0.0);
        bool kept = false;
        if (tid < tot) {
            idx = out_idx[tid];
            v = out_val[tid];
            kept = keep_merged(tid, idx, v);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, kept);
        if ((tid & 31u) == 0) scan[tid >> 5] = (uint32_t)__popc((int)bal);
        __syncthreads();
        uint32_t off = 0;
#pragma unroll
        for (uint32_t w = 0; w < (uint32_t)kThreads / 32u; ++w) {
            const uint32_t c = scan[w];
            off += w < (tid >> 5) ? c : 0u;
            newcount += c;
        }
        if (kept) put(off + (uint32_t)__popc((int)(bal & ((1u << (tid & 31u)) - 1u))), idx, v);
    } else {
        for (uint32_t p = tid; p < tot; p += kThreads) {
            const uint32_t idx = out_idx[p];
            double2 v = out_val[p];
            const bool kept = keep_merged(p, idx, v);
            if (kept) out_val[p] = v;  // (a duplicate's value is read by its head only, and never written)
            keep[p] = kept ? 1u : 0u;
        }
        __syncthreads();
        newcount = block_exclusive_scan(keep, tot, scan);
        for (uint32_t p = tid; p < tot; p += kThreads) {
            const uint32_t pos = keep[p];  // exclusive prefix of the keep flags: kept iff the next differs
            const uint32_t nxt = p + 1 < tot ? keep[p + 1] : newcount;
            if (nxt != pos) put(pos, out_idx[p], out_val[p]);
        }
    }
    if (tid == 0) {
        const bool overflow = newcount > a.zcap;
        if (overflow) a.zflag[s] = 1;
        a.zcount[s] = overflow ? a.zcap : newcount;
        c_n = overflow ? a.zcap : newcount;
        if (last) {
            const uint32_t kept_count = overflow ? a.zcap : newcount;
            a.out_count[s] = kept_count < a.out_cap ? kept_count : a.out_cap;
            int32_t flag = SFFT_OK;
            if (__ldcg(a.zflag + s) || kept_count > a.out_cap)
                flag = SFFT_ERR_CAPACITY;
            else if (s_above > s_kept)
                flag = SFFT_ERR_NOT_CONVERGED;
            a.out_flag[s] = flag;
        }
    }
    return next_ready;
}

// ------------------------------------------------------------------------------------------------
// The decode of a round of a plan whose zhat may hold more than kCarry entries
// ------------------------------------------------------------------------------------------------
// The same steps and the same order of every sum as finish_round's decode, with arrays sized by what
// zhat holds and by what was decoded instead of by their capacities, so that they stay on chip (device
// memory only when they do not fit a.large_smem bytes): the entries' terms lie by bin (stable counting
// split with per-warp counters), the bins are read straight from the round's area, and the candidates
// are sorted by a bitonic network.  Bound by latency (about 40 barriers, 80 with a sort).  Measured with
// gather_owner at n = 2^24, k = 1000, batch 12: 543 us a call, was 1026 (arrays sized by capacity in
// device memory, long bin lists sorted by insertion, one CTA per SM, 140 partial folds per round).
struct LargeLayout {
    size_t e_idx, pre, key, cval, start, slot, s_idx, s_gain, s_t0, s_tf, cnt, out_idx, out_val, keep, scan, total;
};
// nz entries, up to B candidates, tot merged entries; the merge's arrays take the place of the entries'
__host__ __device__ inline LargeLayout large_layout(uint32_t B, uint32_t H, uint32_t nz, uint32_t tot, bool fp64,
                                                    bool val_on_chip) {
    LargeLayout L;
    size_t off = 0;
    const uint32_t P = B < 1024 ? 1024 : B;  // the sort's keys, padded
    L.scan = smem_take(&off, (size_t)(kThreads + 8) * 4);
    L.e_idx = smem_take(&off, (size_t)nz * 4);
    // the decoded bins share their place with the split's counters
    const size_t cnt = nz ? (size_t)split_segments(B) * B * 2 : 0, pre = (size_t)B * 8;
    L.pre = L.cnt = smem_take(&off, pre > cnt ? pre : cnt);
    L.key = smem_take(&off, (size_t)P * 8);
    L.cval = smem_take(&off, val_on_chip ? (size_t)B * 16 : 0);
    const size_t shared = off;
    L.start = smem_take(&off, (size_t)(B + 1) * 4);
    L.slot = smem_take(&off, (size_t)nz * 4);
    L.s_idx = smem_take(&off, (size_t)nz * 4);
    L.s_gain = smem_take(&off, (size_t)nz * 8);
    L.s_t0 = smem_take(&off, (size_t)nz * 16);
    L.s_tf = smem_take(&off, (size_t)nz * H * (fp64 ? 16 : 8));
    const size_t end = off;
    off = shared;
    L.out_idx = smem_take(&off, (size_t)tot * 4);
    L.out_val = smem_take(&off, (size_t)tot * 16);
    L.keep = smem_take(&off, (size_t)(tot + 1) * 4);
    L.total = off > end ? off : end;
    return L;
}
// device-memory slice of a request: the candidates' values, then everything at its largest
size_t exact_large_bytes(uint32_t B, uint32_t H, uint32_t zcap, bool fp64) {
    return (size_t)B * 16 + large_layout(B, H, zcap, zcap + B, fp64, false).total;
}

// whether decode_bin goes beyond its first test on a bin whose subtracted u_0 is u
__device__ __forceinline__ bool worth_decoding(const DecodeCtx& d, float2 u, bool entries) {
    const float m = hypotf(u.x, u.y);
    return m > d.thr_f || (entries && m > d.ref_lo_f && m <= d.ref_hi_f);
}
__device__ __forceinline__ bool worth_decoding(const DecodeCtx& d, double2 u, bool entries) {
    const float f = hypotf((float)u.x, (float)u.y);
    if (d.thr_f > 1e-25f && d.thr_f < 1e25f && f < 1e18f) {  // clear of every bound: as decode_bin_guarded
        if (cmp_guarded(f, d.thr_f) > 0) return true;
        if (cmp_guarded(f, d.thr_f) < 0 && (!entries || cmp_guarded(f, d.ref_hi_f) > 0 || cmp_guarded(f, d.ref_lo_f) < 0))
            return false;
    }
    const double m = cmag(u);
    return m > d.thr || (entries && m > d.ref_lo * d.thr && m <= d.ref_hi * d.thr);
}

// Ascending sort of the nw distinct keys (key holds max(1024, pow2(nw)) words): up to 1024 as four per
// thread, exchanged in registers (strides 1, 2), by shuffles (4 to 64) and through shared memory (128 on:
// 6 exchanges), more by the network in memory.
__device__ __forceinline__ void sort_keys(unsigned long long* key, uint32_t nw) {
    const uint32_t tid = threadIdx.x;
    uint32_t P = 2;
    while (P < nw) P <<= 1;
    if (P <= 4 * (uint32_t)kThreads) {
        unsigned long long k[4];
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) k[q] = 4 * tid + q < nw ? key[4 * tid + q] : ~0ull;
        for (uint32_t size = 2; size <= P; size <<= 1) {
            for (uint32_t stride = size >> 1; stride > 2; stride >>= 1) {
                if (stride >= 128) {
                    __syncthreads();
#pragma unroll
                    for (uint32_t q = 0; q < 4; ++q) key[4 * tid + q] = k[q];
                    __syncthreads();
                }
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q) {
                    const uint32_t i = 4 * tid + q;
                    const unsigned long long o =
                        stride >= 128 ? key[i ^ stride] : __shfl_xor_sync(0xffffffffu, k[q], (int)(stride >> 2));
                    if ((((i & stride) == 0) == ((i & size) == 0)) == (o < k[q])) k[q] = o;
                }
            }
#pragma unroll
            for (uint32_t stride = 2; stride > 0; stride >>= 1)
                if (stride < size)
#pragma unroll
                    for (uint32_t q = 0; q < 4; ++q)
                        if (!(q & stride)) {
                            const unsigned long long x = k[q], y = k[q | stride];
                            const bool up = ((4 * tid + q) & size) == 0;
                            if (up == (x > y)) {
                                k[q] = y;
                                k[q | stride] = x;
                            }
                        }
        }
        __syncthreads();
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (4 * tid + q < nw) key[4 * tid + q] = k[q];
        __syncthreads();
        return;
    }
    for (uint32_t p = nw + tid; p < P; p += kThreads) key[p] = ~0ull;
    __syncthreads();
    for (uint32_t size = 2; size <= P; size <<= 1)
        for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
            for (uint32_t i = tid; i < P / 2; i += kThreads) {
                const uint32_t lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const unsigned long long x = key[lo], y = key[hi];
                if ((lo & size) == 0 ? x > y : x < y) {
                    key[lo] = y;
                    key[hi] = x;
                }
            }
            __syncthreads();
        }
}

template <typename R>
__device__ __forceinline__ bool finish_large(const ExactArgs& a, uint32_t s, uint32_t sigma, uint32_t b,
                                          unsigned char* smem, const uint32_t* next_ctr) {
    using C = typename Cx<R>::T;
    constexpr bool f32 = sizeof(C) == sizeof(float2);
    const uint32_t tid = threadIdx.x, B = a.B, H = a.H;
    __shared__ uint32_t s_nw, s_pre, s_list, s_above, s_kept, s_next_ready;
    __shared__ DecodeCtx d;
    C* area = reinterpret_cast<C*>(a.part) + (size_t)s * a.part_stride;  // the round's bins
    __syncthreads();  // the bins, when this CTA stored them
    if (tid == kThreads - 1) s_next_ready = next_ctr != nullptr && acquire_is(next_ctr, 1u) ? 1u : 0u;
    if (tid == kThreads - 2) fill_ctx_round(d, a, sigma, b);
    if (tid == 0) {
        s_nw = 0;
        s_pre = 0;
        s_list = 0;
        s_above = 0;
        s_kept = 0;
    }
    // zhat is read through L2: in the one-launch path another CTA of this launch may have written it
    uint32_t* zi = a.zidx + (size_t)s * a.zcap;
    double2* zv = a.zval + (size_t)s * a.zcap;
    const uint32_t nz = min(__ldcg(a.zcount + s), a.zcap);
    unsigned char* slice = a.fin_scratch + (size_t)s * a.fin_stride;
    const bool val_on_chip = B <= 512;
    LargeLayout Ly = large_layout(B, H, nz, 0, !f32, val_on_chip);
    unsigned char* mem = smem;
    if (Ly.total > a.large_smem) {
        mem = slice + (size_t)B * 16;
        Ly = large_layout(B, H, a.zcap, a.zcap + B, !f32, false);
    }
    double2* cval = mem == smem && val_on_chip ? reinterpret_cast<double2*>(smem + Ly.cval) : reinterpret_cast<double2*>(slice);
    uint32_t* scan = reinterpret_cast<uint32_t*>(mem + Ly.scan);
    uint32_t* e_idx = reinterpret_cast<uint32_t*>(mem + Ly.e_idx);
    uint2* pre = reinterpret_cast<uint2*>(mem + Ly.pre);
    unsigned long long* key = reinterpret_cast<unsigned long long*>(mem + Ly.key);
    uint32_t* start = reinterpret_cast<uint32_t*>(mem + Ly.start);
    uint32_t* slot = reinterpret_cast<uint32_t*>(mem + Ly.slot);
    uint32_t* s_idx = reinterpret_cast<uint32_t*>(mem + Ly.s_idx);
    double* s_gain = reinterpret_cast<double*>(mem + Ly.s_gain);
    double2* s_t0 = reinterpret_cast<double2*>(mem + Ly.s_t0);
    C* s_tf = reinterpret_cast<C*>(mem + Ly.s_tf);
    // the entries by bin
    const uint32_t Np = (uint32_t)(a.n >> a.logB), logNp = ilog2_u32(Np);
    // (the first four per thread have their gains and values requested here, to arrive during the split)
    double gv[4];
    double2 vv[4];
    for (uint32_t e0 = tid; e0 < nz; e0 += 4 * kThreads) {
        uint32_t iv[4];
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (e0 + q * kThreads < nz) {
                iv[q] = __ldcg(zi + e0 + q * kThreads);
                if (e0 == tid) vv[q] = __ldcg(zv + e0 + q * kThreads);
            }
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (e0 + q * kThreads < nz) {
                e_idx[e0 + q * kThreads] = iv[q];
                uint32_t jb;
                const int32_t o = offset_of((sigma * (iv[q] - b)) & a.nmask, Np, logNp, a.nmask, &jb);
                slot[e0 + q * kThreads] = jb;
                if (e0 == tid) gv[q] = a.wtab[o < 0 ? -o : o];
            }
    }
    __syncthreads();
    const bool next_ready = s_next_ready != 0;
    if (nz != 0)
        split_by_bin(slot, nz, B, reinterpret_cast<uint16_t*>(mem + Ly.cnt), start, scan);
    else
        for (uint32_t j = tid; j <= B; j += kThreads) start[j] = 0;
    // step 4 terms: W(-o(i)) zhat_i w^{a_h sigma i}, as finish_round forms them
    for (uint32_t e0 = tid; e0 < nz; e0 += 4 * kThreads) {
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (e0 != tid && e0 + q * kThreads < nz) {
                uint32_t jb;
                const int32_t o = offset_of((sigma * (e_idx[e0 + q * kThreads] - b)) & a.nmask, Np, logNp, a.nmask, &jb);
                gv[q] = a.wtab[o < 0 ? -o : o];
                vv[q] = __ldcg(zv + e0 + q * kThreads);
            }
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
            if (e0 + q * kThreads >= nz) break;
            const uint32_t i = e_idx[e0 + q * kThreads], at = slot[e0 + q * kThreads];
            s_idx[at] = i;
            s_gain[at] = gv[q];
            const double2 gz = make_double2(gv[q] * vv[q].x, gv[q] * vv[q].y);
            s_t0[at] = gz;  // hashing 0 has offset 0: w^0 = 1
            const float2 g = make_float2((float)gz.x, (float)gz.y);
            const float two_over_n = 2.0f * d.inv_n_f;
            for (uint32_t h = 0; h < H; ++h) {
                const uint32_t ex = (a.a[h] * sigma * i) & a.nmask;
                C w;
                if (f32) {
                    const int32_t es = ex > (a.nmask >> 1) ? (int32_t)((int64_t)ex - (int64_t)a.n) : (int32_t)ex;
                    float sn, cs;
                    sincospif((float)es * two_over_n, &sn, &cs);
                    w.x = g.x * cs + g.y * sn;
                    w.y = g.y * cs - g.x * sn;
                } else {
                    double2 r = gz;
                    if (ex != 0) {
                        const double2 tw = term_root<R>(a, ex);
                        r = make_double2(gz.x * tw.x - gz.y * tw.y, gz.x * tw.y + gz.y * tw.x);
                    }
                    w.x = r.x;
                    w.y = r.y;
                }
                s_tf[at * H + h] = w;
            }
        }
    }
    __syncthreads();
    // the bins that may hold something: above thr (J), or with entries and a residual in the window of a
    // re-estimation.  Their list takes the place of the keys; only they are decoded.
    uint32_t* jl = reinterpret_cast<uint32_t*>(key);
    for (uint32_t b0 = 0; b0 < B; b0 += 4 * kThreads) {  // the same trips for every lane (full-warp ballots)
        const uint32_t j0 = b0 + tid;
        C uv[4];
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (j0 + q * kThreads < B) uv[q] = __ldcg(area + j0 + q * kThreads);
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
            const uint32_t j = j0 + q * kThreads;
            bool want = false;
            if (j < B) {
                C u = uv[q];
                const uint32_t x0 = start[j], x1 = start[j + 1];
                for (uint32_t x = x0; x < x1; ++x) {
                    u.x -= s_tf[x * H].x;
                    u.y -= s_tf[x * H].y;
                }
                want = worth_decoding(d, u, x1 != x0);
            }
            const unsigned mw = __ballot_sync(0xffffffffu, want);
            uint32_t base = 0;
            if ((tid & 31u) == 0 && mw) base = atomicAdd(&s_list, (uint32_t)__popc((int)mw));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (want) jl[base + (uint32_t)__popc((int)(mw & ((1u << (tid & 31u)) - 1u)))] = j;
        }
    }
    __syncthreads();
    // step 4 and the decode, one listed bin per thread
    const uint32_t nlist = s_list;
    for (uint32_t c = tid; c < nlist; c += kThreads) {
        const uint32_t j = jl[c], x0 = start[j], nbin = start[j + 1] - x0;
        C u[kMaxHash];
#pragma unroll
        for (int h = 0; h < kMaxHash; ++h) {
            u[h] = mkc((R)0, (R)0);
            if ((uint32_t)h < H) u[h] = __ldcg(area + (size_t)h * B + j);
        }
        for (uint32_t x = x0; x < x0 + nbin; ++x) {
#pragma unroll
            for (int h = 0; h < kMaxHash; ++h)
                if ((uint32_t)h < H) {
                    u[h].x -= s_tf[x * H + h].x;
                    u[h].y -= s_tf[x * H + h].y;
                }
        }
        // a decoded bin, its gain still to be read: its offset, or the entry re-estimated
        uint32_t where = 0;
        bool above;
        double g0, g1;
        const int kind = decode_bin(d, j, u, RunEntries{nbin}, s_idx + x0, s_gain + x0, &where, &g0, &g1, &above);
        const unsigned m = __activemask();
        const unsigned ma = __ballot_sync(m, above), mw = __ballot_sync(m, kind != 0);
        const uint32_t lane = tid & 31u, leader = (uint32_t)__ffs((int)m) - 1u;
        uint32_t base = 0;
        if (lane == leader) {
            if (ma) atomicAdd(&s_above, (uint32_t)__popc((int)ma));
            if (mw) base = atomicAdd(&s_pre, (uint32_t)__popc((int)mw));
        }
        base = __shfl_sync(m, base, (int)leader);
        if (kind != 0)
            pre[base + (uint32_t)__popc((int)(mw & ((1u << lane) - 1u)))] =
                make_uint2(kind == 1 ? where : x0 + where, j | (kind == 2 ? 0x80000000u : 0u));
    }
    __syncthreads();
    // the decoded bins' gains and values: u_0 in FP64, in the entries' order, times 1 / W(-o) or over W(-o)
    const uint32_t npre = s_pre;
    for (uint32_t c = tid; c < npre; c += kThreads) {
        const uint2 pr = pre[c];
        const uint32_t j = pr.y & 0x7FFFFFFFu;
        const bool known = (pr.y >> 31) != 0;
        const int32_t o = (int32_t)pr.x;
        const uint32_t oa = (uint32_t)(o < 0 ? -o : o);
        const C v = __ldcg(area + j);
        const double gain = known ? s_gain[pr.x] : a.wtab[oa];
        const double ginv = f32 && !known && d.winv ? d.winv[oa] : 0.0;
        const bool kept = known || gain >= d.gmin;
        const unsigned m = __activemask();
        const unsigned mk = __ballot_sync(m, kept && !known), mw = __ballot_sync(m, kept);
        const uint32_t lane = tid & 31u, leader = (uint32_t)__ffs((int)m) - 1u;
        uint32_t base = 0;
        if (lane == leader) {
            if (mk) atomicAdd(&s_kept, (uint32_t)__popc((int)mk));
            if (mw) base = atomicAdd(&s_nw, (uint32_t)__popc((int)mw));
        }
        base = __shfl_sync(m, base, (int)leader);
        if (kept) {
            const uint32_t at = base + (uint32_t)__popc((int)(mw & ((1u << lane) - 1u)));
            double2 u0 = make_double2((double)v.x, (double)v.y);
            for (uint32_t x = start[j]; x < start[j + 1]; ++x) {
                u0.x -= s_t0[x].x;
                u0.y -= s_t0[x].y;
            }
            const uint32_t oi = known ? s_idx[pr.x] : index_at(d, j, o);
            key[at] = ((unsigned long long)oi << 32) | at;
            cval[at] = f32 && !known && d.winv ? make_double2(u0.x * ginv, u0.y * ginv)
                                               : make_double2(u0.x / gain, u0.y / gain);
        }
    }
    __syncthreads();
    const uint32_t nw = s_nw;
    const bool last = a.last_round != 0;
    const uint32_t tot = nz + nw;
    if (mem == smem) {  // the merge's arrays, in place of the entries' where they fit
        Ly = large_layout(B, H, nz, tot, !f32, val_on_chip);
        if (Ly.total > a.large_smem) {
            mem = slice + (size_t)B * 16;
            Ly = large_layout(B, H, a.zcap, a.zcap + B, !f32, false);
        }
    }
    uint32_t* out_idx = reinterpret_cast<uint32_t*>(mem + Ly.out_idx);
    double2* out_val = reinterpret_cast<double2*>(mem + Ly.out_val);
    uint32_t* keep = reinterpret_cast<uint32_t*>(mem + Ly.keep);
    uint32_t newcount = nz;
    if (nw == 0) {
        // nothing decoded: zhat stays as it is
        if (last)
            for (uint32_t e = tid; e < nz && e < a.out_cap; e += kThreads) {
                a.out_idx[(size_t)s * a.out_cap + e] = e_idx[e];
                a.out_val[(size_t)s * a.out_cap + e] = __ldcg(zv + e);
            }
    } else {
        // the candidates by index (distinct: a decode lies in its own bin)
        if (nw <= (uint32_t)kThreads) {
            unsigned long long k = 0;
            uint32_t r = 0;
            if (tid < nw) {
                k = key[tid];
                for (uint32_t q = 0; q < nw; ++q) r += key[q] < k ? 1u : 0u;
            }
            __syncthreads();
            if (tid < nw) key[r] = k;
            __syncthreads();
        } else {
            sort_keys(key, nw);
        }
        // merge what into zhat (zhat first on equal indices), then drop entries below prune * thr
        for (uint32_t e = tid; e < nz; e += kThreads) {
            const unsigned long long k = (unsigned long long)e_idx[e] << 32;
            uint32_t lo = 0, hi = nw;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (key[mid] < k) lo = mid + 1; else hi = mid;
            }
            out_idx[e + lo] = e_idx[e];
            out_val[e + lo] = __ldcg(zv + e);
        }
        for (uint32_t c = tid; c < nw; c += kThreads) {
            const uint32_t idx = (uint32_t)(key[c] >> 32);
            const uint32_t pos = c + upper_bound_u32(e_idx, nz, idx);
            out_idx[pos] = idx;
            out_val[pos] = cval[(uint32_t)key[c]];
        }
        __syncthreads();
        for (uint32_t p = tid; p < tot; p += kThreads) {
            uint32_t kp = 0;
            const uint32_t idx = out_idx[p];
            if (p == 0 || out_idx[p - 1] != idx) {
                double2 v = out_val[p];
                if (p + 1 < tot && out_idx[p + 1] == idx) {
                    v.x += out_val[p + 1].x;
                    v.y += out_val[p + 1].y;
                    out_val[p] = v;  // the duplicate at p + 1 is never a head and is not written
                }
                if (f32)
                    kp = hypotf((float)v.x, (float)v.y) < a.drop_f ? 0u : 1u;
                else
                    kp = dropped(v, a) ? 0u : 1u;
            }
            keep[p] = kp;
        }
        __syncthreads();
        newcount = block_exclusive_scan(keep, tot, scan);
        for (uint32_t p = tid; p < tot; p += kThreads) {
            const uint32_t pos = keep[p];
            const uint32_t nxt = p + 1 < tot ? keep[p + 1] : newcount;
            if (nxt == pos) continue;
            const uint32_t idx = out_idx[p];
            const double2 v = out_val[p];
            if (pos < a.zcap) {
                zi[pos] = idx;
                zv[pos] = v;
            }
            if (last && pos < a.out_cap) {
                a.out_idx[(size_t)s * a.out_cap + pos] = idx;
                a.out_val[(size_t)s * a.out_cap + pos] = v;
            }
        }
    }
    if (tid == 0) {
        const bool overflow = newcount > a.zcap;
        const uint32_t count = overflow ? a.zcap : newcount;
        if (overflow) a.zflag[s] = 1;
        if (nw != 0) a.zcount[s] = count;
        if (last) {
            a.out_count[s] = count < a.out_cap ? count : a.out_cap;
            int32_t flag = SFFT_OK;
            if (__ldcg(a.zflag + s) || count > a.out_cap)
                flag = SFFT_ERR_CAPACITY;
            else if (s_above > s_kept)
                flag = SFFT_ERR_NOT_CONVERGED;
            a.out_flag[s] = flag;
        }
    }
    return next_ready;
}

#ifndef SFFT_ROUND_MIN_BLOCKS
#define SFFT_ROUND_MIN_BLOCKS 2  // resident CTAs per SM the register budget is sized for
#endif

template <typename R>
__global__ void __launch_bounds__(kThreads, SFFT_ROUND_MIN_BLOCKS) k_exact_round(const ExactArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t s = a.req_base + blockIdx.y, c = blockIdx.x;
    const ReqView rq = req_view(a.reqs, a.x, a.n * sizeof(typename Cx<R>::T), a.seed, s, a.nmask);
    const uint32_t sigma = a.e_sigma, b = a.e_b;
    gather_fold<R>(a, rq.x, rq.xmask, s, c, sigma, b, smem);
    // arrival: the last CTA of request s finishes the round (nobody waits)
    if (arrive(a.counter + s, a.chunks) == 0) return;
    finish_round<R>(a, s, sigma, b, a.fin_scratch ? a.fin_scratch + (size_t)s * a.fin_stride : smem);
    if (threadIdx.x == 0) a.counter[s] = 0;
}

// ------------------------------------------------------------------------------------------------
// One launch per batch: all rounds' chunks, finishers chained by arrival counters
// ------------------------------------------------------------------------------------------------
// The decodes of request s from round t on, in this CTA, for as long as the next round's bins have
// arrived.  Round t > 0's decode is the second of two arrivals at its counter2 (its bins, round t - 1's
// decode); round 0's needs no zhat and follows its bins here.  Each decode also reads the next round's
// counter2 (an acquire load that overlaps its own loads): when those bins have arrived, this chain is
// the last party of that round and goes on without an arrival of its own.  (seed, id) name the
// request's draws.
template <typename R, int NR, int KIND>
__device__ __forceinline__ void decode_chain(const StepParams<NR>& sp, uint32_t t, const ExactArgs* a, uint32_t s,
                                             uint64_t seed, uint32_t id, uint32_t sigma, uint32_t b,
                                             unsigned char* smem) {
    if (t > 0 && arrive_pair(a->counter2 + s) == 0) return;
    bool bins_here = true;  // the bins just formed are in this CTA's shared memory
    for (bool carried = false;; carried = true) {
        const uint32_t* next_ctr = t + 1 < sp.R ? sp.r[t + 1].counter2 + s : nullptr;
        const bool next_ready =
            KIND == kDecodeLarge ? finish_large<R>(*a, s, sigma, b, smem, next_ctr)
                  : finish_round<R, KIND>(*a, s, sigma, b, smem, kFinDecode, carried, bins_here, next_ctr);
        if (threadIdx.x == 0) a->counter2[s] = 0;  // both arrivals of round t have happened (or none, t = 0)
        if (t + 1 >= sp.R) break;
        a = &sp.r[++t];
        bins_here = false;
        // zhat of round t - 1 is published by the arrival at round t's second counter (which also
        // orders this round's shared-memory writes, the kept zhat among them, before the next reads)
        if (next_ready)
            __syncthreads();
        else if (arrive_pair(a->counter2 + s) == 0)
            break;
        exact_hash(seed, id, t, a->nmask, &sigma, &b);
    }
}

template <typename R, int NR, int KIND>
__global__ void __launch_bounds__(kThreads, SFFT_ROUND_MIN_BLOCKS) k_exact_step(const __grid_constant__ StepParams<NR> sp) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t tid = threadIdx.x;
    uint32_t t = 0;
    while (t + 1 < sp.R && blockIdx.x >= sp.seg[t + 1]) ++t;
    const ExactArgs* a = &sp.r[t];
    const uint32_t local = blockIdx.x - sp.seg[t];
    const uint32_t c = local % a->gctas;
    const uint32_t s = a->req_base + local / a->gctas;
    const ReqView rq = req_view(a->reqs, a->x, a->n * sizeof(typename Cx<R>::T), a->seed, s, a->nmask);
    uint32_t sigma, b;
    exact_hash(rq.seed, rq.id, t, a->nmask, &sigma, &b);
    if (KIND == kDecodeLarge && a->owner)
        gather_owner<R>(*a, rq.x, rq.xmask, s, c, sigma, b, smem);
    else
        gather_fold<R>(*a, rq.x, rq.xmask, s, c, sigma, b, smem);
    if (arrive(a->counter + s, a->gctas) == 0) return;
    // the round's bins, in this CTA's shared memory (the gather's staging area holds H B values)
    finish_round<R, KIND>(*a, s, sigma, b, smem, kFinBins);
    if (tid == 0) a->counter[s] = 0;  // every chunk of round t has arrived
    decode_chain<R, NR, KIND>(sp, t, a, s, rq.seed, rq.id, sigma, b, smem);
}

// ------------------------------------------------------------------------------------------------
// Multi-channel batches with shared hashing (see ChanParams)
// ------------------------------------------------------------------------------------------------
// Gather and fold: CTA (t, rho, c) sums, for each hashing h of round t and every channel, the terms
// G_{s + a_h} w^{sigma b (s + a_h)} x_{sigma s} over the samples s = s0 + i, i = rho' + j B (rho' the
// first index of residue class rho), j in chunk c: bin rho of hashing h.  Warp 0 issues one bulk copy
// per row (C contiguous complex values) into shared memory, then forms the rows' coefficients (one
// row per lane) while the copies are in flight; once they have landed, thread ch folds channel ch in
// row order.
constexpr uint32_t kChanWaitLimit = 1u << 22;  // tries of a bounded wait (3.8 us each: 16 s)
// Every thread of a CTA: whether the copies that complete phase 0 of `bar` have landed, within `limit` tries.
// If not (never expected), *error is set, and the copies get a second bounded wait, to end while their
// shared memory is still this CTA's.
__device__ __forceinline__ bool copies_landed(uint64_t* bar, uint32_t limit, uint32_t* error) {
    if (mbar_wait(bar, 0, limit)) return true;
    if (threadIdx.x == 0) atomicExch(error, 1u);
    mbar_wait(bar, 0, limit);
    return false;
}
template <int NR>
__global__ void __launch_bounds__(kThreads) k_chan_gather(const __grid_constant__ ChanParams<NR> cp) {
    extern __shared__ __align__(16) unsigned char smem[];  // bulk copies need 16-byte alignment
    __shared__ __align__(8) uint64_t bar;
    const uint32_t C = cp.C, tid = threadIdx.x;
    float2* rows = reinterpret_cast<float2*>(smem);                                       // [kChanRows][C]
    float2* coef = reinterpret_cast<float2*>(smem + (size_t)kChanRows * C * sizeof(float2));  // [kChanRows][kMaxHash]
    uint32_t t = 0;
    while (t + 1 < cp.R && blockIdx.x >= cp.cseg[t + 1]) ++t;
    const ExactArgs& a = cp.r[t];
    const uint32_t local = blockIdx.x - cp.cseg[t];
    const uint32_t rho = local & (a.B - 1), c = local / a.B;
    const int64_t s0 = -a.T - (int64_t)a.maxshift;
    const uint32_t cnt = (uint32_t)(2 * a.T + 1) + a.maxshift;
    const uint32_t i_first = (rho - (uint32_t)s0) & (a.B - 1);
    const uint32_t nrows = i_first < cnt ? (cnt - 1 - i_first) / a.B + 1 : 0;
    const uint32_t j_beg = c * kChanRows;
    const uint32_t m = nrows > j_beg ? min(kChanRows, nrows - j_beg) : 0u;  // rows of this chunk
    if (tid == 0) mbar_init(&bar, 1);
    __syncthreads();
    if (tid < 32) {
        uint32_t sigma, b;
        exact_hash(cp.seed, cp.id, t, a.nmask, &sigma, &b);
        const uint32_t sb = sigma * b;
        const bool ok = tid < m;
        const int32_t sl = (int32_t)(s0 + (int64_t)i_first + (int64_t)(j_beg + tid) * a.B);
        // the copies first, the coefficients while they are in flight
        if (tid == 0) mbar_arrive_expect_tx(&bar, m * C * (uint32_t)sizeof(float2));
        __syncwarp();
        if (ok) {
            const uint32_t row = (sigma * (uint32_t)sl) & a.nmask;
            bulk_copy_g2s(rows + (size_t)tid * C, static_cast<const float2*>(cp.x) + (size_t)row * C,
                          C * (uint32_t)sizeof(float2), &bar);
        }
#pragma unroll
        for (int h = 0; h < kMaxHash; ++h) {
            float2 co = make_float2(0.0f, 0.0f);
            const int32_t th = sl + (int32_t)a.a[h];
            if ((uint32_t)h < a.H && ok && th >= -a.T && th <= a.T) {
                const float gt = a.taps32[th < 0 ? -th : th];
                const uint32_t e = (sb * (uint32_t)th) & a.nmask;
                const int32_t es = e > (a.nmask >> 1) ? (int32_t)((int64_t)e - (int64_t)a.n) : (int32_t)e;
                float sn, cs;
                sincospif((float)es * (2.0f / (float)a.n), &sn, &cs);
                co = make_float2(gt * cs, -gt * sn);
            }
            if (tid < kChanRows) coef[tid * kMaxHash + h] = co;
        }
    }
    __syncthreads();  // the coefficients
    if (!copies_landed(&bar, kChanWaitLimit, cp.error)) return;  // (the partial sums stay as they are)
    for (uint32_t ch = tid; ch < C; ch += kThreads) {
        float2 acc[kMaxHash];
#pragma unroll
        for (int h = 0; h < kMaxHash; ++h) acc[h] = make_float2(0.0f, 0.0f);
        for (uint32_t j = 0; j < m; ++j) {
            const float2 v = rows[(size_t)j * C + ch];
#pragma unroll
            for (int h = 0; h < kMaxHash; ++h) acc[h] = cfma(coef[j * kMaxHash + h], v, acc[h]);
        }
        float2* area = static_cast<float2*>(a.part) + (size_t)ch * a.part_stride;
#pragma unroll
        for (int h = 0; h < kMaxHash; ++h)
            if ((uint32_t)h < a.H) area[((size_t)c * a.H + h) * a.B + rho] = acc[h];
    }
}

// The bins of every (round, slot) at once: partial folds summed in chunk order, bit-reversed, B-point
// FFT, left at the start of the slot's area of the round.  Bound by L2 reads and latency: four CTAs per SM
// (64 registers, shared memory for the bins alone) instead of two took 256 channels at n = 2^21 from 102 to
// 98 us a call.
template <int NR>
__global__ void __launch_bounds__(kThreads, 4) k_chan_bins(const __grid_constant__ StepParams<NR> sp,
                                                                              uint64_t seed, uint32_t id) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t t = 0;
    while (t + 1 < sp.R && blockIdx.x >= sp.seg[t + 1]) ++t;
    const ExactArgs& a = sp.r[t];
    const uint32_t s = blockIdx.x - sp.seg[t];
    uint32_t sigma, b;
    exact_hash(seed, id, t, a.nmask, &sigma, &b);
    finish_round<float>(a, s, sigma, b, smem, kFinBins);
}

// The decodes: one CTA per channel slot runs them in round order (zhat of round t feeds round t + 1).
// If the gather flagged a copy that never landed, every slot reports SFFT_ERR_TIMEOUT instead.
template <int NR, int KIND>
__global__ void __launch_bounds__(kThreads, SFFT_ROUND_MIN_BLOCKS) k_chan_decode(const __grid_constant__ StepParams<NR> sp,
                                                                                uint64_t seed, uint32_t id,
                                                                                const uint32_t* error) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t s = blockIdx.x;
    if (*error) {
        if (threadIdx.x == 0) {
            const ExactArgs& a = sp.r[sp.R - 1];
            a.out_count[s] = 0;
            a.out_flag[s] = SFFT_ERR_TIMEOUT;
        }
        return;
    }
    for (uint32_t t = 0; t < sp.R; ++t) {
        const ExactArgs& a = sp.r[t];
        uint32_t sigma, b;
        exact_hash(seed, id, t, a.nmask, &sigma, &b);
        if (KIND == kDecodeLarge)
            finish_large<float>(a, s, sigma, b, smem, nullptr);
        else
            finish_round<float, KIND>(a, s, sigma, b, smem, kFinDecode, t > 0);
        __syncthreads();  // zhat of round t is read by round t + 1 (same CTA)
    }
}

// ------------------------------------------------------------------------------------------------
// Mixed batches: requests of different plans in one launch
// ------------------------------------------------------------------------------------------------
// The scheme of k_exact_step over requests that each have their own plan: the gathers of every round of
// every request are in the grid from the start, round by round (segment i = the CTAs of one (round,
// request)), the decodes are chained by arrival counters and nothing waits.  A round's argument block
// comes from device memory, its per-request fields are pointed at the request's own workspace.  Against
// the device queue it replaces, where a request's next round was gathered only after the last one's
// decode: 408 us, was 870 (96 requests of six plans, n = 2^16 .. 2^22).
template <typename R, int KIND>
__global__ void __launch_bounds__(kThreads, SFFT_ROUND_MIN_BLOCKS) k_exact_batch(const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) ExactArgs sa;
    const uint32_t tid = threadIdx.x;
    // the segment of this CTA: the last whose first CTA is not above it, kThreads probes at a time
    uint32_t lo = 0, len = ba.nseg;
    while (len > 1) {
        const uint32_t stride = (len + kThreads - 1) / kThreads, i = tid * stride;
        const uint32_t n = (uint32_t)__syncthreads_count(i < len && ba.seg[lo + i] <= blockIdx.x);
        lo += (n - 1) * stride;
        len = min(stride, len - (n - 1) * stride);
    }
    const uint32_t c = blockIdx.x - ba.seg[lo], who = ba.seg_who[lo];
    const uint32_t r = who & 0xFFFFFFu;
    uint32_t t = who >> 24;
    uint32_t* const counters = ba.counter + (size_t)r * 2 * kMaxRounds;  // per round; then the second ones
    const uint32_t rounds = ba.req_rounds[r];
    auto load_round = [&](uint32_t round) {
        __syncthreads();  // every reader of the block is done
        const uint32_t* src = reinterpret_cast<const uint32_t*>(ba.rdesc + ba.req_rd0[r] + round);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&sa);
        for (uint32_t w = tid; w < sizeof(ExactArgs) / 4; w += kThreads) dst[w] = src[w];
        __syncthreads();
        if (tid == 0) {
            sa.reqs = ba.reqs + r;
            sa.req_base = 0;
            sa.part = ba.part + (size_t)r * ba.part_stride + sa.part_bytes;
            sa.part_stride = 0;
            sa.counter = counters + round;
            sa.counter2 = counters + kMaxRounds + round;
            sa.zidx = ba.zidx + (size_t)r * ba.z_stride;
            sa.zval = ba.zval + (size_t)r * ba.z_stride;
            sa.zcount = ba.zcount + r;
            sa.zflag = ba.zflag + r;
            sa.fin_scratch = ba.fin + (size_t)r * ba.fin_stride;
            sa.fin_stride = 0;
            sa.out_idx = ba.out_idx + (size_t)r * ba.out_cap;
            sa.out_val = ba.out_val + (size_t)r * ba.out_cap;
            sa.out_cap = ba.out_cap;
            sa.out_count = ba.out_count + r;
            sa.out_flag = ba.out_flag + r;
        }
        __syncthreads();
    };
    load_round(t);
    const ReqView rq = req_view(sa.reqs, nullptr, 0, 0, 0, sa.nmask);
    uint32_t sigma, b;
    exact_hash(rq.seed, rq.id, t, sa.nmask, &sigma, &b);
    if (KIND == kDecodeLarge && sa.owner)
        gather_owner<R>(sa, rq.x, rq.xmask, 0, c, sigma, b, smem);
    else
        gather_fold<R>(sa, rq.x, rq.xmask, 0, c, sigma, b, smem);
    if (arrive(sa.counter, sa.gctas) == 0) return;
    finish_round<R, KIND>(sa, 0, sigma, b, smem, kFinBins);
    if (tid == 0) *sa.counter = 0;
    if (t > 0 && arrive_pair(sa.counter2) == 0) return;
    // the decodes from round t on (as decode_chain)
    for (bool first = true;; first = false) {
        const uint32_t* next_ctr = t + 1 < rounds ? counters + kMaxRounds + t + 1 : nullptr;
        const bool next_ready = KIND == kDecodeLarge
                                    ? finish_large<R>(sa, 0, sigma, b, smem, next_ctr)
                                    : finish_round<R, KIND>(sa, 0, sigma, b, smem, kFinDecode, !first, first, next_ctr);
        if (tid == 0) *sa.counter2 = 0;
        if (++t >= rounds) break;
        if (!next_ready && arrive_pair(counters + kMaxRounds + t) == 0) break;
        load_round(t);
        exact_hash(rq.seed, rq.id, t, sa.nmask, &sigma, &b);
    }
}

template <typename R>
static void launch_batch(const BatchArgs& a, uint32_t ctas, size_t smem, cudaStream_t st, int kind) {
    if (kind == kDecodeLarge)
        k_exact_batch<R, kDecodeLarge><<<ctas, kThreads, smem, st>>>(a);
    else if (kind == kDecodeMasks)
        k_exact_batch<R, kDecodeMasks><<<ctas, kThreads, smem, st>>>(a);
    else
        k_exact_batch<R, kDecodeLists><<<ctas, kThreads, smem, st>>>(a);
}
cudaError_t launch_exact_batch(const BatchArgs& a, uint32_t ctas, size_t smem, cudaStream_t st, bool fp64, int kind) {
    if (ctas == 0) return cudaSuccess;
    if (fp64)
        launch_batch<double>(a, ctas, smem, st, kind);
    else
        launch_batch<float>(a, ctas, smem, st, kind);
    return cudaGetLastError();
}

// The gather's wait where no copy ever lands: a barrier whose phase nothing completes.
constexpr uint32_t kWaitCheckLimit = 1u << 17;  // half a second, twice
__global__ void __launch_bounds__(kThreads) k_chan_wait_check(uint32_t limit, uint32_t* error) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    copies_landed(&bar, limit, error);
}
cudaError_t launch_chan_wait_check(uint32_t* error, cudaStream_t st) {
    k_chan_wait_check<<<1, kThreads, 0, st>>>(kWaitCheckLimit, error);
    return cudaGetLastError();
}
// What the decodes of a channel batch report once the gather has set *error (which the caller has seen set:
// there are no bins to decode).
cudaError_t launch_chan_timeouts(const uint32_t* error, uint32_t slots, uint32_t* count, int32_t* flag, cudaStream_t st) {
    StepParams<8> sp = {};
    sp.R = 1;
    sp.r[0].out_count = count;
    sp.r[0].out_flag = flag;
    k_chan_decode<8, kDecodeMasks><<<slots, kThreads, 0, st>>>(sp, 0, 0, error);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// decode on caller bins (single CTA)
// ------------------------------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(kThreads) k_exact_decode(const DecodeArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_nw, s_above, s_kept;
    const uint32_t tid = threadIdx.x, B = a.B;
    const uint32_t zcap = a.nz > 0 ? a.nz : 1;
    const FinLayout Ly = fin_layout(B, a.H, zcap, 16);
    double2* U = reinterpret_cast<double2*>(smem + Ly.U);
    uint32_t* ent_idx = reinterpret_cast<uint32_t*>(smem + Ly.ent_idx);
    uint32_t* ent_bin = reinterpret_cast<uint32_t*>(smem + Ly.ent_bin);
    double* ent_gain = reinterpret_cast<double*>(smem + Ly.ent_gain);
    uint32_t* bin_cnt = reinterpret_cast<uint32_t*>(smem + Ly.bin_cnt);
    uint32_t* bin_start = reinterpret_cast<uint32_t*>(smem + Ly.bin_start);
    uint32_t* bin_list = reinterpret_cast<uint32_t*>(smem + Ly.bin_list);
    uint32_t* cand_idx = reinterpret_cast<uint32_t*>(smem + Ly.cand_idx);
    double2* cand_val = reinterpret_cast<double2*>(smem + Ly.cand_val);
    uint32_t* srt_idx = reinterpret_cast<uint32_t*>(smem + Ly.srt_idx);
    double2* srt_val = reinterpret_cast<double2*>(smem + Ly.srt_val);
    uint32_t* scan = reinterpret_cast<uint32_t*>(smem + Ly.scan);
    __shared__ DecodeCtx d;
    if (tid == 0)
        fill_ctx(d, a.n, a.nmask, B, a.logB, a.H, a.shift64, a.sigma, a.b, a.wtab, a.thr, a.iso_tol, a.gmin, a.ref_lo,
                 a.ref_hi, a.ref_tol);
    __syncthreads();
    for (uint32_t i = tid; i < a.H * B; i += kThreads) U[i] = a.u[i];
    for (uint32_t e = tid; e < a.nz; e += kThreads) {
        const uint32_t i = a.zidx[e];
        ent_idx[e] = i;
        uint32_t jb;
        const int32_t o = offset_of((a.sigma * (i - a.b)) & a.nmask, d, &jb);
        ent_bin[e] = jb;
        ent_gain[e] = a.wtab[o < 0 ? -o : o];
    }
    if (tid == 0) {
        s_nw = 0;
        s_above = 0;
        s_kept = 0;
    }
    __syncthreads();
    bucket_entries(ent_bin, a.nz, B, bin_cnt, bin_start, bin_list, scan);
    for (uint32_t j = tid; j < B; j += kThreads) {
        using C = typename Cx<R>::T;
        C u[kMaxHash];  // the caller's bins, in the precision of the decisions
        for (uint32_t h = 0; h < a.H; ++h) {
            u[h].x = U[h * B + j].x;
            u[h].y = U[h * B + j].y;
        }
        uint32_t oi = 0;
        double gain = 1.0, ginv;  // this decode divides by the gain (its context has no 1 / W table)
        bool above;
        const int kind = decode_bin(d, j, u, ListEntries{bin_list + bin_start[j], bin_start[j + 1] - bin_start[j]}, ent_idx,
                                    ent_gain, &oi, &gain, &ginv, &above);
        if (above) atomicAdd(&s_above, 1u);
        if (kind == 1) atomicAdd(&s_kept, 1u);
        if (kind != 0) {
            const uint32_t slot = atomicAdd(&s_nw, 1u);
            cand_idx[slot] = oi;
            cand_val[slot] = make_double2(U[j].x / gain, U[j].y / gain);
        }
    }
    __syncthreads();
    const uint32_t nw = s_nw;
    rank_sort(cand_idx, cand_val, nw, srt_idx, srt_val);
    for (uint32_t p = tid; p < nw; p += kThreads) {
        a.widx[p] = srt_idx[p];
        a.wval[p] = srt_val[p];
    }
    if (tid == 0) {
        *a.count = nw;
        *a.nabove = s_above;
        *a.nkept = s_kept;
    }
}

__global__ void k_philox(uint32_t k0, uint32_t k1, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t count,
                         uint32_t* out) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const Words4 w = philox4x32_10(c0, c1, c2, c3 + i, k0, k1);
    for (int q = 0; q < 4; ++q) out[4 * (size_t)i + q] = w.w[q];
}

// ------------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------------
// The dynamic shared-memory ceiling of a kernel is process-wide: it is only ever raised, so a plan
// created later with smaller rounds cannot lower it under another plan's feet.
template <int NR>
static cudaError_t launch_chan_nr(const ExactArgs* rounds, uint32_t R, uint32_t C, const void* x, uint64_t seed,
                                  uint32_t id, size_t smem, uint32_t* error, cudaStream_t st, cudaEvent_t before,
                                  cudaEvent_t after) {
    ChanParams<NR> cp;
    StepParams<NR> sp;
    cp.R = sp.R = R;
    cp.C = C;
    cp.seed = seed;
    cp.id = id;
    cp.x = x;
    cp.error = error;
    cp.cseg[0] = 0;
    sp.seg[0] = 0;
    for (uint32_t t = 0; t < R; ++t) {
        const uint64_t w = (uint64_t)cp.cseg[t] + (uint64_t)rounds[t].chunks * rounds[t].B;
        if (w > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
        cp.cseg[t + 1] = (uint32_t)w;
        sp.seg[t + 1] = sp.seg[t] + C;
        cp.r[t] = sp.r[t] = rounds[t];
    }
    const size_t gsmem = (size_t)kChanRows * C * sizeof(float2) + (size_t)kChanRows * kMaxHash * sizeof(float2);
    static std::mutex mu;
    static size_t set_to = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (set_to < kChanRows * kChanMaxC * sizeof(float2) + kChanRows * kMaxHash * sizeof(float2)) {
            const int full = (int)(kChanRows * kChanMaxC * sizeof(float2) + kChanRows * kMaxHash * sizeof(float2));
            cudaError_t e = cudaFuncSetAttribute(k_chan_gather<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, full);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_chan_gather<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, full);
            if (e != cudaSuccess) return e;
            set_to = (size_t)full;
        }
    }
    cudaError_t e = cudaMemsetAsync(error, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    if (before && (e = cudaEventRecord(before, st)) != cudaSuccess) return e;
    k_chan_gather<NR><<<cp.cseg[R], kThreads, gsmem, st>>>(cp);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (after && (e = cudaEventRecord(after, st)) != cudaSuccess) return e;
    size_t bsmem = 0;  // the bins alone: four CTAs per SM
    for (uint32_t t = 0; t < R; ++t) bsmem = std::max(bsmem, (size_t)rounds[t].H * rounds[t].B * sizeof(float2));
    k_chan_bins<NR><<<sp.seg[R], kThreads, bsmem, st>>>(sp, seed, id);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (rounds[0].kind == kDecodeLarge)
        k_chan_decode<NR, kDecodeLarge><<<C, kThreads, smem, st>>>(sp, seed, id, error);
    else if (rounds[0].kind == kDecodeMasks)
        k_chan_decode<NR, kDecodeMasks><<<C, kThreads, smem, st>>>(sp, seed, id, error);
    else
        k_chan_decode<NR, kDecodeLists><<<C, kThreads, smem, st>>>(sp, seed, id, error);
    return cudaGetLastError();
}

cudaError_t launch_exact_channels(const ExactArgs* rounds, uint32_t R, uint32_t C, const void* x, uint64_t seed,
                                  uint32_t id, size_t smem, uint32_t* error, cudaStream_t st, cudaEvent_t before,
                                  cudaEvent_t after) {
    if (R == 0 || R > kMaxRounds || C == 0 || C % 32 || C > kChanMaxC || !error) return cudaErrorInvalidValue;
    if (R <= 8) return launch_chan_nr<8>(rounds, R, C, x, seed, id, smem, error, st, before, after);
    return launch_chan_nr<32>(rounds, R, C, x, seed, id, smem, error, st, before, after);
}

template <typename R, int KIND>
static cudaError_t raise_exact_smem(size_t bytes, size_t* cur) {
    if (bytes <= *cur) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    auto raise = [&](const void* kernel) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    raise((const void*)k_exact_step<R, 8, KIND>);
    raise((const void*)k_exact_step<R, 32, KIND>);
    if constexpr (sizeof(R) == sizeof(float)) {
        raise((const void*)k_chan_decode<8, KIND>);
        raise((const void*)k_chan_decode<32, KIND>);
    }
    if (e == cudaSuccess) *cur = bytes;
    return e;
}
template <typename R>
static cudaError_t raise_exact_smem(size_t bytes, int kind, size_t* limits) {
    if (kind == kDecodeLarge) return raise_exact_smem<R, kDecodeLarge>(bytes, limits + kind);
    if (kind == kDecodeMasks) return raise_exact_smem<R, kDecodeMasks>(bytes, limits + kind);
    return raise_exact_smem<R, kDecodeLists>(bytes, limits + kind);
}
// the kernels that serve every kind of plan
cudaError_t set_round_smem_limit(size_t bytes, bool fp64) {
    static std::mutex mu;  // plans may be created from several threads
    std::lock_guard<std::mutex> lk(mu);
    static size_t limit[2] = {0, 0};
    size_t& cur = limit[fp64 ? 1 : 0];
    if (bytes <= cur) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    auto raise = [&](const void* kernel) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    if (fp64) {
        raise((const void*)k_exact_round<double>);
    } else {
        raise((const void*)k_exact_round<float>);
        raise((const void*)k_chan_bins<8>);
        raise((const void*)k_chan_bins<32>);
    }
    if (e == cudaSuccess) cur = bytes;
    return e;
}
cudaError_t set_exact_smem_limit(size_t bytes, bool fp64, int kind) {
    const cudaError_t e = set_round_smem_limit(bytes, fp64);
    if (e != cudaSuccess) return e;
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    static size_t limit[2][3] = {{0, 0, 0}, {0, 0, 0}};
    return fp64 ? raise_exact_smem<double>(bytes, kind, limit[1]) : raise_exact_smem<float>(bytes, kind, limit[0]);
}
cudaError_t set_batch_smem_limit(size_t bytes, bool fp64, int kind) {
    static std::mutex mu;
    std::lock_guard<std::mutex> lk(mu);
    static size_t limit[2][3] = {{0, 0, 0}, {0, 0, 0}};
    size_t& cur = limit[fp64 ? 1 : 0][kind];
    if (bytes <= cur) return cudaSuccess;
    const void* kernels[2][3] = {
        {(const void*)k_exact_batch<float, 0>, (const void*)k_exact_batch<float, 1>, (const void*)k_exact_batch<float, 2>},
        {(const void*)k_exact_batch<double, 0>, (const void*)k_exact_batch<double, 1>, (const void*)k_exact_batch<double, 2>}};
    const cudaError_t e =
        cudaFuncSetAttribute(kernels[fp64 ? 1 : 0][kind], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) cur = bytes;
    return e;
}

cudaError_t launch_exact_round(const ExactArgs& a, uint32_t batch, size_t smem, cudaStream_t st, bool fp64) {
    const dim3 grid(a.chunks, batch);
    if (fp64)
        k_exact_round<double><<<grid, kThreads, smem, st>>>(a);
    else
        k_exact_round<float><<<grid, kThreads, smem, st>>>(a);
    return cudaGetLastError();
}

template <int NR, int KIND>
static void launch_step_kind(const StepParams<NR>& sp, uint32_t ctas, size_t smem, cudaStream_t st, bool fp64) {
    if (fp64)
        k_exact_step<double, NR, KIND><<<ctas, kThreads, smem, st>>>(sp);
    else
        k_exact_step<float, NR, KIND><<<ctas, kThreads, smem, st>>>(sp);
}
template <int NR>
static void launch_step(const StepParams<NR>& sp, uint32_t ctas, size_t smem, cudaStream_t st, bool fp64, int kind) {
    if (kind == kDecodeLarge)
        launch_step_kind<NR, kDecodeLarge>(sp, ctas, smem, st, fp64);
    else if (kind == kDecodeMasks)
        launch_step_kind<NR, kDecodeMasks>(sp, ctas, smem, st, fp64);
    else
        launch_step_kind<NR, kDecodeLists>(sp, ctas, smem, st, fp64);
}
template <int NR>
static cudaError_t launch_step_nr(const ExactArgs* rounds, uint32_t R, uint32_t batch, size_t smem, cudaStream_t st,
                                  bool fp64) {
    StepParams<NR> sp;
    sp.R = R;
    sp.seg[0] = 0;
    for (uint32_t t = 0; t < R; ++t) {
        const uint64_t end = (uint64_t)sp.seg[t] + (uint64_t)rounds[t].gctas * batch;
        if (end > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;  // grid limit
        sp.seg[t + 1] = (uint32_t)end;
        sp.r[t] = rounds[t];
    }
    const uint32_t ctas = sp.seg[R];
    if (ctas == 0) return cudaSuccess;
    launch_step<NR>(sp, ctas, smem, st, fp64, (int)rounds[0].kind);  // one kind for the whole plan
    return cudaGetLastError();
}

cudaError_t launch_exact_step(const ExactArgs* rounds, uint32_t R, uint32_t batch, size_t smem, cudaStream_t st,
                              bool fp64) {
    if (R == 0 || R > kMaxRounds) return cudaErrorInvalidValue;
    if (R <= 8) return launch_step_nr<8>(rounds, R, batch, smem, st, fp64);
    return launch_step_nr<32>(rounds, R, batch, smem, st, fp64);
}

cudaError_t launch_exact_decode(const DecodeArgs& a, cudaStream_t st) {
    const size_t smem = fin_layout(a.B, a.H, a.nz > 0 ? a.nz : 1, 16).total;
    cudaError_t e;
    if (a.fp64) {
        e = cudaFuncSetAttribute(k_exact_decode<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_exact_decode<double><<<1, kThreads, smem, st>>>(a);
    } else {
        e = cudaFuncSetAttribute(k_exact_decode<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_exact_decode<float><<<1, kThreads, smem, st>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_philox(uint32_t k0, uint32_t k1, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                          uint32_t count, uint32_t* out, cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    k_philox<<<(count + 255) / 256, 256, 0, st>>>(k0, k1, c0, c1, c2, c3, count, out);
    return cudaGetLastError();
}

}  // namespace sfft
