// mf_filter.cuh -- the fused sources and sinks of the bank filter, shared by
// the per-batch kernels (mf_filter.cu) and the persistent scheduler
// (mf_persist.cu).
#pragma once
#include "mf_passes.cuh"

namespace mf {

// ---------------------------------------------------------------------------
// FP64 anchors.  psi(k) = C0 + sum_p c_p u^p, u = (k df)^(-1/3), in turns.  With
// w_p = c_p u^p the k-derivatives are
//   d^n psi/dk^n = (-1)^n sum_p [p (p+3) ... (p+3(n-1)) / 3^n] w_p / k^n,
// so the Taylor coefficients at the anchor centre k_a = g D + D/2 are
//   q1 = -sum p w_p / (3k),  q2 = sum p(p+3) w_p / (18 k^2),
//   q3 = -sum p(p+3)(p+6) w_p / (162 k^3),  q4 = sum p(p+3)(p+6)(p+9) w_p / (1944 k^4).
// psi mod 1 and q1 (which multiplies offsets up to D/2) are formed in FP64 --
// u from an FP32 seed and one FP64 Newton step u <- u (4 - f u^3) / 3 -- and
// q2..q4 in FP32.  Record: float4 (psi mod 1, q1, q2, q3) and float q4.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void anchor_record(double c1, double c2, double c3, double c5, int64_t g, int log2D,
                                              double df, float4 &rec, float &rec4) {
    const int64_t ka = (g << log2D) + ((1 << log2D) >> 1);
    const double f = (double)ka * df;
    double uu = (double)rcbrtf((float)f);
    uu = uu * (4.0 - f * uu * uu * uu) * (1.0 / 3.0);
    const double u2 = uu * uu;
    const double psi = -0.125 + uu * (c1 + uu * (c2 + uu * (c3 + u2 * c5)));
    const double S1 = uu * (c1 + uu * (2.0 * c2 + uu * (3.0 * c3 + u2 * (5.0 * c5))));
    const double ik = df * u2 * uu;   // 1 / k_a
    const double r0 = psi - rint(psi);
    const float uf = (float)uu, ikf = (float)ik;
    const float w1 = (float)c1 * uf, w2 = (float)c2 * uf * uf, w3 = (float)c3 * uf * uf * uf;
    const float w5 = (float)c5 * (uf * uf) * (uf * uf * uf);
    const float S2 = 4.f * w1 + 10.f * w2 + 18.f * w3 + 40.f * w5;
    const float S3 = 28.f * w1 + 80.f * w2 + 162.f * w3 + 440.f * w5;
    const float S4 = 280.f * w1 + 880.f * w2 + 1944.f * w3 + 6160.f * w5;
    const float ik2 = ikf * ikf;
    rec = make_float4((float)r0, (float)(-S1 * ik * (1.0 / 3.0)), S2 * ik2 * (1.f / 18.f),
                      -S3 * ik2 * ikf * (1.f / 162.f));
    rec4 = S4 * ik2 * ik2 * (1.f / 1944.f);
}

// Smallest k in [a, c] with P[k] - P0 >= target, or c (P does not decrease), by
// one warp: 32 probes a step, so four dependent loads for 2^19 bins instead of
// twenty.  All lanes call it with the same arguments and get the result.
__device__ __forceinline__ int64_t edge_search(const double *P, double P0, double target, int64_t a, int64_t c, int lane) {
    while (a < c) {
        const int64_t step = (c - a + 31) / 32;
        const int64_t k = a + lane * step;
        const bool reach = k < c && P[k] - P0 >= target;
        const unsigned m = __ballot_sync(0xffffffffu, reach);
        if (m) {   // the first probe that reaches it
            const int first = __ffs(m) - 1;
            c = a + first * step;
            if (first > 0) a = c - step + 1;
        } else {   // none of the probes below c: past the last one
            a += ((c - 1 - a) / step) * step + 1;
        }
    }
    return a;
}

// ---------------------------------------------------------------------------
// pass-1 source: X_k = W_k e^{-i Psi_k} on the band, 0 elsewhere; k >= N/2 is
// always outside (one-sided spectrum), so the upper half of every column is 0.
// ---------------------------------------------------------------------------
template <int L, int C, int LG1>
struct TemplateSrc {
    static constexpr bool kHalfZero = true;
    static constexpr bool kSplitTw = true;   // same rounding as the persistent pass 1
    // one anchor record (float4 + float) per non-zero column row, staged per tile
    static constexpr size_t kScratchBytes = (size_t)(L / 2) * (sizeof(float4) + sizeof(float));
    struct Params {
        const float2 *W;
        const UnitInfo *units;
        const float4 *anchors;
        const float *anchors4;
        int anc_stride, log2D;
        int anc_slots;   // > 0: several bands share a template's anchors, slot mod anc_slots
    };
    const Params &p;
    const int tile, unit, slot;
    float4 *sa;
    float *sa4;
    unsigned *rel = nullptr;   // deferred release (persistent scheduler), done by thread 0 once loads are in flight
    __device__ TemplateSrc(const Params &pp, int tl, int un, int sl, void *scratch)
        : p(pp), tile(tl), unit(un), slot(sl), sa((float4 *)scratch), sa4((float *)((float4 *)scratch + L / 2)) {}
    // All C L/32 threads of the tile call load() (it contains a block barrier).
    __device__ __forceinline__ void load(int seq, int t, float2 *v) const {
        constexpr int T = L / 32;
        const UnitInfo u = p.units[unit];
        const int aslot = p.anc_slots > 0 ? slot % p.anc_slots : slot;
        const float4 *anc0 = p.anchors + (int64_t)aslot * p.anc_stride;   // index: anchor_slot_index(g)
        const float *anc40 = p.anchors4 + (int64_t)aslot * p.anc_stride;
        constexpr int LGL = cx_ilog2(L);
        const int k1 = tile * C + seq;
        const int D = 1 << p.log2D;
        float2 w[16];
        bool in[16];
        const int k0 = k1 + (t << LG1);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int k = k0 + ((r * T) << LG1);
            in[r] = (k >= u.k_lo) && (k < u.k_hi);
            w[r] = in[r] ? __ldg(&p.W[k]) : czero();   // no load outside the band
        }
        if (D >= C && p.log2D <= LG1) {
            // Every column of this tile falls in the same anchor group on a
            // given row n, so the tile needs one anchor per row:
            // g(n) = (tile C >> log2D) + n (N1 >> log2D), record (tile C >> log2D) R + n,
            // staged once in shared memory.
            const int gstep = 1 << (LG1 - p.log2D);
            const int gcol = (tile * C) >> p.log2D;
            const int gbase = gcol - u.g_lo;
            const float4 *acol = anc0 + ((int64_t)gcol << (LGL - 1));
            const float *acol4 = anc40 + ((int64_t)gcol << (LGL - 1));
            for (int n = threadIdx.x; n < L / 2; n += C * T) {
                const int a = gbase + n * gstep;
                if (a >= 0 && a < u.n_anc &&
                    MF_DBG(((int64_t)gcol << (LGL - 1)) + n < p.anc_stride, kDbgAnchor)) {
                    sa[n] = __ldcg(&acol[n]);   // anchors may be rewritten in the same launch (ring)
                    sa4[n] = __ldcg(&acol4[n]);
                }
            }
            release_hook(rel);
            __syncthreads();
            // offset from the anchor centre is the same on every row (D divides N1)
            const float d = (float)((k1 & (D - 1)) - (D >> 1));
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int n = t + r * T;
                float2 x = czero();
                if (__any_sync(0xffffffffu, in[r])) {   // rows outside the band of the whole warp cost nothing
                    const float4 a = sa[n];
                    const float a4 = sa4[n];
                    float ph = fmaf(fmaf(fmaf(fmaf(a4, d, a.w), d, a.z), d, a.y), d, a.x);
                    ph -= rintf(ph);
                    float sn, cs;
                    __sincosf(6.283185307179586f * ph, &sn, &cs);
                    x = make_float2(fmaf(w[r].x, cs, w[r].y * sn), fmaf(w[r].y, cs, -w[r].x * sn));  // W e^{-i 2 pi ph}
                }
                v[r] = in[r] ? x : czero();
            }
        } else {
            // Several anchor groups per row of the tile (short segments): each
            // element reads its record.  The records of four rows are loaded
            // before the first is used: a row at a time, one after the other
            // behind its test, is 16 trips to L2 a tile (16 templates at N =
            // 2^16, D = 16, all tiles resident: 11.1 us, 9.4 so).
            release_hook(rel);
            const int half = D >> 1;
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
                if (!__any_sync(0xffffffffu, in[c] || in[c + 1] || in[c + 2] || in[c + 3])) {
#pragma unroll
                    for (int r = c; r < c + 4; ++r) v[r] = czero();
                    continue;
                }
                float4 a[4];
                float a4[4], d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = k0 + (((c + i) * T) << LG1);
                    const int kk = in[c + i] ? k : u.k_lo;
                    const int g = kk >> p.log2D;
                    int64_t ai = anchor_slot_index(g, LGL + LG1, LG1, p.log2D);
                    if (!MF_DBG(ai >= 0 && ai < p.anc_stride, kDbgAnchor)) ai = 0;
                    a[i] = __ldcg(&anc0[ai]);
                    a4[i] = __ldcg(&anc40[ai]);
                    d[i] = (float)(kk - ((g << p.log2D) + half));
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = c + i;
                    float ph = fmaf(fmaf(fmaf(fmaf(a4[i], d[i], a[i].w), d[i], a[i].z), d[i], a[i].y), d[i], a[i].x);
                    ph -= rintf(ph);
                    float sn, cs;
                    __sincosf(6.283185307179586f * ph, &sn, &cs);
                    const float2 x = make_float2(fmaf(w[r].x, cs, w[r].y * sn), fmaf(w[r].y, cs, -w[r].x * sn));
                    v[r] = in[r] ? x : czero();
                }
            }
        }
    }
};

// The same for bands of a few rows per column (the chi^2 sub-bands): where no
// lane of a warp holds more than one row of the band, each lane forms its one
// element and the first stage is dft32_single, as in the narrow form of the
// staged pass 1.  16 templates at N = 2^16, p = 16: 46 us without, 40 here.
template <int L, int C, int LG1>
struct TemplateSrcNarrow : TemplateSrc<L, C, LG1> {
    using Base = TemplateSrc<L, C, LG1>;
    using typename Base::Params;
    mutable bool single = false;
    mutable int rs = 0;
    __device__ TemplateSrcNarrow(const Params &pp, int tl, int un, int sl, void *scratch)
        : Base(pp, tl, un, sl, scratch) {}
    __device__ __forceinline__ void load(int seq, int t, float2 *v) const {
        constexpr int T = L / 32, LGL = cx_ilog2(L), LGS = cx_ilog2(T) + LG1;   // row step N / 32 bins
        const Params &p = this->p;
        const int4 band = __ldg(reinterpret_cast<const int4 *>(p.units + this->unit));   // k_lo, k_hi, ..
        const int k0 = this->tile * C + seq + (t << LG1);
        const int rlo = band.x <= k0 ? 0 : min(16, (band.x - k0 + (1 << LGS) - 1) >> LGS);
        const int rhi = band.y <= k0 ? 0 : min(16, (band.y - k0 + (1 << LGS) - 1) >> LGS);
        // a block-wide choice: load() of the general form holds a barrier
        if (__syncthreads_or(rhi - rlo > 1)) {
            Base::load(seq, t, v);
            return;
        }
        single = true;
        rs = min(rlo, 15);
        v[0] = czero();
        if (rhi > rlo) {
            const int k = k0 + (rlo << LGS), g = k >> p.log2D;
            int64_t ai = anchor_slot_index(g, LGL + LG1, LG1, p.log2D);
            if (!MF_DBG(ai >= 0 && ai < p.anc_stride, kDbgAnchor)) ai = 0;
            ai += (int64_t)(p.anc_slots > 0 ? this->slot % p.anc_slots : this->slot) * p.anc_stride;
            const float2 w = __ldg(&p.W[k]);
            const float4 a = __ldcg(&p.anchors[ai]);
            const float a4 = __ldcg(&p.anchors4[ai]);
            const float d = (float)(k - ((g << p.log2D) + ((1 << p.log2D) >> 1)));
            float ph = fmaf(fmaf(fmaf(fmaf(a4, d, a.w), d, a.z), d, a.y), d, a.x);
            ph -= rintf(ph);
            float sn, cs;
            __sincosf(6.283185307179586f * ph, &sn, &cs);
            v[0] = make_float2(fmaf(w.x, cs, w.y * sn), fmaf(w.y, cs, -w.x * sn));
        }
    }
};

// ---------------------------------------------------------------------------
// MF_PHASE_FP64: the phase at 64-bit accuracy at every bin.  GB300 issues two
// FP64 operations per SM and clock, so psi in FP64 at every bin (27 of them
// with the unused derivatives) was two thirds of the filter's time: 1125 of
// 1714 us for 250 templates at N = 2^18.  Between FP64 anchors the phase is
// instead summed in turns mod 1 as 64-bit fixed point: with the integer offset
// d from the anchor centre,
//   psi = r0 + d (q1 + d (q2 + d q3))  (mod 1, exact in 2^-64 turns)  +  d^4 (q4 + d (q5 + d (q6 + d q7)))
// where the cubic part is three 64-bit integer multiply-adds (d is an integer,
// so the coefficients count mod 1) and the small rest FP32.  anchor_log2D64
// bounds what is left out and the size of the FP32 part: the sum, in 2^-32
// turns, is off by 2^-33 (the low word, rounded) + 2^-33 (the FP32 part in those
// units) + its own rounding, 1e-10, + 5e-11 left out: 4e-10 turns at most.
// u comes from a step of third order, u (1 + e/3 + 2 e^2/9) with e = 1 - f u^3,
// as many operations as a Newton step, which leaves 4e-14 of u, up to 4e-10 turns
// of a light template at 10 Hz.  What counts is the phase the sincos gets.  psi in
// FP64 at every bin, rounded to FP32 in [-1/2, 1/2], is off by up to 1.5e-8
// turns; half turns are taken off first here (they change signs only), so the
// rounding is 2^-27 at most and the whole 7.9e-9.  Over 1-34 solar masses, 10 to
// 40 Hz, N = 2^10 .. 2^22: 7.7e-9 and 3.3e-9 rms; FP64 at every bin 1.5e-8 and
// 6.5e-9.  The distance of the z series from 64 bits, 2^14 .. 2^20, is 0.4 to
// 1.3 % below that of FP64 at every bin (sincos and FFT make up most of it).
// Record: three planes of 16 bytes (r0, q1 | q2, q3 | q4, q5, q6, q7), r0 with
// the half unit that rounds the low word.
// ---------------------------------------------------------------------------
struct Anchor64 {
    unsigned long long r0, q1, q2, q3;
    float q4, q5, q6, q7;
};
// x mod 1 in 2^-64 turns: the sum with 1.5 * 2^(52 - 30) leaves x in units of
// 2^-30 in the mantissa, and the rest of x is exact (a conversion from FP64 to
// a 64-bit integer is several FP64 operations)
__device__ __forceinline__ unsigned long long turns_fixed(double x) {
    x -= rint(x);
    constexpr double kBig = 6291456.0;   // 1.5 * 2^22
    const double s = x + kBig;
    const long long hi = __double_as_longlong(s) & ((1ll << 30) - 1);   // x mod 1 in 2^-30 turns
    const double rest = x - (s - kBig);                                  // |rest| <= 2^-31
    const float top = (float)rest;                                       // rest to 2^-55
    return ((unsigned long long)hi << 34) + (unsigned long long)(long long)__float2ll_rn(top * 1.8446744073709552e19f);
}
__device__ __forceinline__ Anchor64 anchor_record64(double c1, double c2, double c3, double c5, int64_t g, int log2D,
                                                    double df) {
    const int64_t ka = (g << log2D) + ((1 << log2D) >> 1);
    const double f = (double)ka * df;
    double uu = (double)rcbrtf((float)f);
    const double e = fma(-f, uu * uu * uu, 1.0);
    uu = fma(uu, e * fma(e, 2.0 / 9.0, 1.0 / 3.0), uu);
    const double u2 = uu * uu;
    const double psi = -0.125 + uu * (c1 + uu * (c2 + uu * (c3 + u2 * c5)));
    const double S1 = uu * (c1 + uu * (2.0 * c2 + uu * (3.0 * c3 + u2 * (5.0 * c5))));
    const double S2 = uu * (4.0 * c1 + uu * (10.0 * c2 + uu * (18.0 * c3 + u2 * (40.0 * c5))));
    const double ik = df * u2 * uu;   // 1 / k_a
    const double ik2 = ik * ik;
    const float uf = (float)uu, ikf = (float)ik, ik4 = (ikf * ikf) * (ikf * ikf);
    const float w1 = (float)c1 * uf, w2 = (float)c2 * uf * uf, w3 = (float)c3 * uf * uf * uf;
    const float w5 = (float)c5 * (uf * uf) * (uf * uf * uf);
    const double S3 = uu * (28.0 * c1 + uu * (80.0 * c2 + uu * (162.0 * c3 + u2 * (440.0 * c5))));
    Anchor64 a;
    a.r0 = turns_fixed(psi) + (1ull << 31);
    a.q1 = turns_fixed(S1 * ik * (-1.0 / 3.0));
    a.q2 = turns_fixed(S2 * ik2 * (1.0 / 18.0));
    a.q3 = turns_fixed(S3 * (ik2 * ik) * (-1.0 / 162.0));
    a.q4 = (280.f * w1 + 880.f * w2 + 1944.f * w3 + 6160.f * w5) * ik4 * (1.f / 1944.f);
    a.q5 = -(3640.f * w1 + 12320.f * w2 + 29160.f * w3 + 104720.f * w5) * ik4 * ikf * (1.f / 29160.f);
    a.q6 = (58240.f * w1 + 209440.f * w2 + 524880.f * w3 + 2094400.f * w5) * ik4 * (ikf * ikf) * (1.f / 524880.f);
    a.q7 = -(1106560.f * w1 + 4188800.f * w2 + 11022480.f * w3 + 48171200.f * w5) * ik4 * (ikf * ikf * ikf) *
           (1.f / 11022480.f);
    return a;
}
// phase in turns at integer offset d, d4 = d^4, less the half turn that sign
// says (bit 31: it belongs on the sine and the cosine): in [-1/4, 1/4]
__device__ __forceinline__ float anchor_phase64(const float4 &p0, const float4 &p1, const float4 &p2, int d, float df,
                                                float d4, unsigned &sign) {
    auto word = [](float lo, float hi) {
        return ((unsigned long long)(unsigned)__float_as_int(hi) << 32) | (unsigned)__float_as_int(lo);
    };
    const unsigned long long dd = (unsigned long long)(long long)d;
    const unsigned long long t =
        word(p0.x, p0.y) + dd * (word(p0.z, p0.w) + dd * (word(p1.x, p1.y) + dd * word(p1.z, p1.w)));
    const float tail = d4 * fmaf(df, fmaf(df, fmaf(df, p2.w, p2.z), p2.y), p2.x);
    // |tail| < 2^-10: added to 1.5 * 2^-9 its mantissa counts 2^-32 turns
    const unsigned hi = (unsigned)(t >> 32) + (unsigned)(__float_as_int(tail + 0.0029296875f) - 0x3b400000);
    const int rest = (int)(hi << 1) >> 1;   // mod half a turn
    sign = (hi ^ (unsigned)rest) & 0x80000000u;
    return (float)rest * 2.3283064365386963e-10f;   // 2^-32; rounded once
}
__device__ __forceinline__ float flip_sign(float x, unsigned sign) { return __int_as_float(__float_as_int(x) ^ (int)sign); }

// pass-1 source of MF_PHASE_FP64
template <int L, int C, int LG1>
struct TemplateSrc64 {
    static constexpr bool kHalfZero = true;
    static constexpr bool kSplitTw = true;
    static constexpr size_t kScratchBytes = (size_t)(L / 2) * 3 * sizeof(float4);
    struct Params {
        const float2 *W;
        const UnitInfo *units;
        const float4 *anchors;   // slot: three planes of anc_stride records
        int anc_stride, log2D, anc_slots;
    };
    const Params &p;
    const int tile, unit, slot;
    float4 *sa;
    __device__ TemplateSrc64(const Params &pp, int tl, int un, int sl, void *scratch)
        : p(pp), tile(tl), unit(un), slot(sl), sa((float4 *)scratch) {}
    // All C L/32 threads of the tile call load() (it contains a block barrier).
    __device__ __forceinline__ void load(int seq, int t, float2 *v) const {
        constexpr int T = L / 32;
        constexpr int LGL = cx_ilog2(L);
        const UnitInfo u = p.units[unit];
        const int aslot = p.anc_slots > 0 ? slot % p.anc_slots : slot;
        const float4 *anc = p.anchors + (int64_t)aslot * 3 * p.anc_stride;   // index: anchor_slot_index(g)
        const int k1 = tile * C + seq;
        const int D = 1 << p.log2D;
        const int k0 = k1 + (t << LG1);
        float2 w[16];
        bool in[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int k = k0 + ((r * T) << LG1);
            in[r] = (k >= u.k_lo) && (k < u.k_hi);
            w[r] = in[r] ? __ldg(&p.W[k]) : czero();   // no load outside the band
        }
        const bool shared_row = D >= C && p.log2D <= LG1;   // one record per column row, as in TemplateSrc
        if (shared_row) {
            const int gstep = 1 << (LG1 - p.log2D);
            const int gcol = (tile * C) >> p.log2D;
            const int gbase = gcol - u.g_lo;
            const float4 *acol = anc + ((int64_t)gcol << (LGL - 1));
            for (int n = threadIdx.x; n < L / 2; n += C * T) {
                const int a = gbase + n * gstep;
                if (a >= 0 && a < u.n_anc && MF_DBG(((int64_t)gcol << (LGL - 1)) + n < p.anc_stride, kDbgAnchor)) {
#pragma unroll
                    for (int h = 0; h < 3; ++h) sa[h * (L / 2) + n] = __ldcg(&acol[(int64_t)h * p.anc_stride + n]);
                }
            }
            __syncthreads();
        }
        const int d0 = (k1 & (D - 1)) - (D >> 1);   // the same on every row when D divides N1
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            if (!__any_sync(0xffffffffu, in[r])) {
                v[r] = czero();
                continue;
            }
            float4 a0, a1, a2;
            int d = d0;
            if (shared_row) {
                const int n = t + r * T;
                a0 = sa[n];
                a1 = sa[L / 2 + n];
                a2 = sa[L + n];
            } else {
                const int k = k0 + ((r * T) << LG1);
                const int kk = in[r] ? k : u.k_lo;
                const int g = kk >> p.log2D;
                int64_t ai = anchor_slot_index(g, LGL + LG1, LG1, p.log2D);
                if (!MF_DBG(ai >= 0 && ai < p.anc_stride, kDbgAnchor)) ai = 0;
                a0 = __ldcg(&anc[ai]);
                a1 = __ldcg(&anc[ai + p.anc_stride]);
                a2 = __ldcg(&anc[ai + 2 * (int64_t)p.anc_stride]);
                d = kk - ((g << p.log2D) + (D >> 1));
            }
            const float df = (float)d;
            unsigned sign;
            const float ph = anchor_phase64(a0, a1, a2, d, df, (df * df) * (df * df), sign);
            float sn, cs;
            __sincosf(6.283185307179586f * ph, &sn, &cs);
            sn = flip_sign(sn, sign);
            cs = flip_sign(cs, sign);
            const float2 x = make_float2(fmaf(w[r].x, cs, w[r].y * sn), fmaf(w[r].y, cs, -w[r].x * sn));
            v[r] = in[r] ? x : czero();   // rows outside the band read stale records
        }
    }
};

// FP32-only phase (precision-sweep reference): psi evaluated directly in FP32.
template <int L, int C, int LG1>
struct TemplateSrcF32 {
    static constexpr bool kHalfZero = true;
    static constexpr bool kSplitTw = true;
    struct Params {
        const float2 *W;
        const UnitInfo *units;
        const double *tmpl;
        float df;
    };
    static constexpr size_t kScratchBytes = 0;
    const Params &p;
    const int tile, unit;
    __device__ TemplateSrcF32(const Params &pp, int tl, int un, int, void *) : p(pp), tile(tl), unit(un) {}
    __device__ __forceinline__ void load(int seq, int t, float2 *v) const {
        constexpr int T = L / 32;
        const UnitInfo u = p.units[unit];
        const double *Tm = p.tmpl + (int64_t)u.tmpl * kTmplStride;
        const float c1 = (float)Tm[TF_C1], c2 = (float)Tm[TF_C2], c3 = (float)Tm[TF_C3], c5 = (float)Tm[TF_C5];
        const int k1 = tile * C + seq;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int k = k1 + ((t + r * T) << LG1);
            const bool in = (k >= u.k_lo) && (k < u.k_hi);
            const int kk = in ? k : u.k_lo;
            const float2 w = __ldg(&p.W[kk]);
            const float uu = rcbrtf((float)kk * p.df);
            const float u2 = uu * uu;
            float ph = -0.125f + uu * (c1 + uu * (c2 + uu * (c3 + u2 * c5)));
            ph -= rintf(ph);
            float s, c;
            __sincosf(6.283185307179586f * ph, &s, &c);
            const float2 x = make_float2(fmaf(w.x, c, w.y * s), fmaf(w.y, c, -w.x * s));
            v[r] = in ? x : czero();
        }
    }
};

// ---------------------------------------------------------------------------
// pass-2 sink: rho epilogue.  raw_j = row FFT output at j = j2 + N2 j1;
// rho_j = |raw_j| rho_scale.  Tracks the argmax (lowest j on ties) and
// appends every j with |raw_j|^2 > thr2.
// ---------------------------------------------------------------------------
// max(0, a[0], ..., a[R-1]) (NaNs ignored, as by fmaxf) by pairwise halving:
// a dependency chain of log2 R instead of R.
template <int R>
__device__ __forceinline__ float tree_max0(const float *a) {
    if constexpr (R == 1) {
        return fmaxf(0.f, a[0]);
    } else {
        float h[(R + 1) / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) h[i] = fmaxf(a[i], a[i + R / 2]);
        if constexpr (R % 2) h[R / 2] = a[R - 1];
        return tree_max0<(R + 1) / 2>(h);
    }
}

template <int L, int C>
struct RhoSink {
    struct Params {
        const UnitInfo *units;
        float4 *partials;
        mf_trigger *staged;
        uint64_t *keys;
        unsigned long long *counter;
        int64_t cap;
        int log2N2, nblk, seg_idx;
        KeyLayout kl;
    };
    const Params &p;
    const int tile, unit;
    UnitInfo u;
    float bp;
    int bj;
    float2 bz;
    __device__ RhoSink(const Params &pp, int tl, int un, int)
        : p(pp), tile(tl), unit(un), bp(-1.f), bj(0x7fffffff), bz(make_float2(0.f, 0.f)) {
        u = p.units[un];
    }
    template <int R>
    __device__ __forceinline__ void store(int seq, int b, int stride, const float2 *v) {
        const int j2 = tile * C + seq;
        float pw[R];
#pragma unroll
        for (int r = 0; r < R; ++r) pw[r] = fmaf(v[r].x, v[r].x, v[r].y * v[r].y);
        const float m = tree_max0<R>(pw);
        // The butterfly's outputs j2 + N2 (b + r stride) increase with r, so its
        // argmax with the lowest-j tie rule is the first r with pw[r] == m.
        if (m >= bp) {
            int rs = R - 1;
#pragma unroll
            for (int r = R - 2; r >= 0; --r) rs = (pw[r] == m) ? r : rs;
            const int j = j2 + ((b + rs * stride) << p.log2N2);
            if (m > bp || j < bj) {
                float2 z = v[R - 1];
#pragma unroll
                for (int r = R - 2; r >= 0; --r) z = (r == rs) ? v[r] : z;
                bp = m;
                bj = j;
                bz = z;
            }
        }
        if (__any_sync(0xffffffffu, m > u.thr2)) {
            const int lane = threadIdx.x & 31;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool pred = pw[r] > u.thr2;
                const unsigned msk = __ballot_sync(0xffffffffu, pred);
                if (msk == 0u) continue;   // warp-uniform
                const int leader = __ffs(msk) - 1;
                unsigned long long base = 0ull;
                if (lane == leader) base = atomicAdd(p.counter, (unsigned long long)__popc(msk));
                base = __shfl_sync(0xffffffffu, base, leader);
                if (pred) {
                    const unsigned long long slot = base + (unsigned long long)__popc(msk & ((1u << lane) - 1u));
                    if (slot < (unsigned long long)p.cap &&
                        MF_DBG(j2 + ((b + r * stride) << p.log2N2) < (1 << p.kl.j_bits), kDbgOut)) {
                        const int j = j2 + ((b + r * stride) << p.log2N2);
                        mf_trigger tr;
                        tr.tmpl = u.tmpl;
                        tr.seg = p.seg_idx;
                        tr.j = j;
                        tr.rho = sqrtf(pw[r]) * u.rho_scale;
                        tr.z_re = v[r].x * u.z_scale;
                        tr.z_im = v[r].y * u.z_scale;
                        p.staged[slot] = tr;
                        p.keys[slot] = ((uint64_t)u.tmpl << (p.kl.seg_bits + p.kl.j_bits)) |
                                       ((uint64_t)p.seg_idx << p.kl.j_bits) | (uint64_t)j;
                    }
                }
            }
        }
    }
    // CTA argmax -> partials[unit * nblk + tile]
    __device__ __forceinline__ void finish(float2 *smem) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float op = __shfl_xor_sync(0xffffffffu, bp, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            const float ox = __shfl_xor_sync(0xffffffffu, bz.x, o);
            const float oy = __shfl_xor_sync(0xffffffffu, bz.y, o);
            if (op > bp || (op == bp && oj < bj)) { bp = op; bj = oj; bz = make_float2(ox, oy); }
        }
        __syncthreads();   // the last FFT stage may still be reading shared memory
        float4 *red = reinterpret_cast<float4 *>(smem);
        if (lane == 0) red[warp] = make_float4(bp, __int_as_float(bj), bz.x, bz.y);
        __syncthreads();
        if (threadIdx.x == 0) {
            constexpr int nw = C * (L / 32) / 32;
            float4 best = red[0];
            for (int w = 1; w < nw; ++w) {
                const float4 c = red[w];
                const int cj = __float_as_int(c.y), bjj = __float_as_int(best.y);
                if (c.x > best.x || (c.x == best.x && cj < bjj)) best = c;
            }
            p.partials[(int64_t)unit * p.nblk + tile] = best;
        }
    }
};

// ---------------------------------------------------------------------------
// per-unit set-up and peaks
// ---------------------------------------------------------------------------
// Unit of template t: band, scale factors, threshold, anchor range.
__device__ __forceinline__ UnitInfo unit_info(const SegDev &seg, const double *T, int t, double f_low, float thr, int log2D) {
    const double N = (double)seg.N, fs = seg.fs;
    const double fisco = T[TF_FISCO];
    const double fc = fisco < 0.5 * fs ? fisco : 0.5 * fs;
    int64_t lo = (int64_t)ceil(f_low * N / fs);
    int64_t hi = (int64_t)floor(fc * N / fs) + 1;
    if (lo < 1) lo = 1;
    if (hi > seg.N / 2) hi = seg.N / 2;
    if (hi < lo) hi = lo;
    const double Q = seg.P[hi] - seg.P[lo];              // sum_band f^(-7/3)/S  (Eq. 4 / (4 df A^2))
    const double rs = sqrt(seg.consts->P_tot / Q);
    UnitInfo u;
    u.k_lo = (int32_t)lo;
    u.k_hi = (int32_t)hi;
    u.g_lo = (int32_t)(lo >> log2D);
    u.n_anc = (int32_t)(((hi - 1) >> log2D) - (lo >> log2D) + 1);
    u.rho_scale = (float)rs;
    const double th = (double)thr / rs;
    u.thr2 = (float)(th * th);
    u.z_scale = (float)(4.0 * seg.df * T[TF_AMP] / seg.consts->alpha);
    u.tmpl = t;
    return u;
}

// the call's control words, zeroed by the first kernel of the call (one block
// of it calls this; a memset would be one more launch)
__device__ __forceinline__ void clear_ctl(FilterCtl *ctl) {
    unsigned *w = reinterpret_cast<unsigned *>(ctl);
    for (unsigned i = threadIdx.x; i < sizeof(FilterCtl) / 4; i += blockDim.x) w[i] = 0u;
}

// the anchor records of one unit, blocks bx of nbx
__device__ __forceinline__ void unit_anchors(const SegDev &seg, const double *T, const UnitInfo &u, int log2D,
                                             int max_anc, float4 *out, float *out4, int reps, int64_t rep_stride,
                                             int bx, int nbx) {
    const double c1 = T[TF_C1], c2 = T[TF_C2], c3 = T[TF_C3], c5 = T[TF_C5];
    for (int i = bx * blockDim.x + threadIdx.x; i < u.n_anc; i += nbx * blockDim.x) {
        float4 r;
        float r4;
        const int64_t g = (int64_t)u.g_lo + i;
        anchor_record(c1, c2, c3, c5, g, log2D, seg.df, r, r4);
        const int64_t a = anchor_slot_index(g, seg.log2N, seg.log2N1, log2D);
        if (!MF_DBG(a >= 0 && a < max_anc, kDbgAnchor)) continue;
        for (int k = 0; k < reps; ++k) {
            out[a + k * rep_stride] = r;
            out4[a + k * rep_stride] = r4;
        }
    }
}

// The peak of one unit from its pass-2 partials, by one warp: the loudest
// sample, the first of equal ones.
__device__ __forceinline__ void unit_peak(const UnitInfo &u, int n_all, const float4 *pp, int nblk, int seg_idx,
                                          int n_seg, mf_peak *peaks) {
    const int lane = threadIdx.x & 31;
    float bp = -1.f;
    int bj = 0x7fffffff;
    float bx = 0.f, by = 0.f;
    for (int i = lane; i < nblk; i += 32) {
        const float4 c = pp[i];
        const int cj = __float_as_int(c.y);
        if (c.x > bp || (c.x == bp && cj < bj)) { bp = c.x; bj = cj; bx = c.z; by = c.w; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float op = __shfl_xor_sync(0xffffffffu, bp, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        const float ox = __shfl_xor_sync(0xffffffffu, bx, o);
        const float oy = __shfl_xor_sync(0xffffffffu, by, o);
        if (op > bp || (op == bp && oj < bj)) { bp = op; bj = oj; bx = ox; by = oy; }
    }
    if (lane == 0) {
        mf_peak pk;
        pk.rho = sqrtf(bp) * u.rho_scale;
        pk.j = bj;
        pk.z_re = bx * u.z_scale;
        pk.z_im = by * u.z_scale;
        if (MF_DBG(u.tmpl >= 0 && u.tmpl < n_all && seg_idx < n_seg, kDbgOut))
            peaks[(int64_t)u.tmpl * n_seg + seg_idx] = pk;
    }
}

}  // namespace mf
