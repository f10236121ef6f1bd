// mf_filter.cu -- the hot path of the bank filter (Eqs. 1, 3, 4 of
// arXiv:0906.4175): per (template, segment) unit
//   k_units    band [k_lo, k_hi) (Sec. 1.1 band rule), sigma from the FP64
//              prefix table, rho and z scale factors, anchor range;
//   k_anchors  the 2PN phase Psi/(2 pi) in FP64 at anchor bins, reduced mod 1,
//              plus its first four k-derivatives (FP32 Taylor coefficients);
//              k_anchors64 the records of MF_PHASE_FP64;
//   pass 1     template generation h~_k = e^{-i Psi_k} in registers (FP32
//              quartic Taylor from the nearest anchor, __sincosf of the reduced
//              phase), weighting by W_k = f^(-7/6) conj(s~_k)/S_k, column IFFTs,
//              four-step twiddle, one complex64 exchange write;
//   pass 2     row IFFTs and the rho epilogue: |z|^2 threshold test, argmax with
//              lowest-j tie-break, warp-aggregated trigger append;
//   k_reduce_peaks / k_sort_triggers   deterministic peaks and (tmpl, seg, j)
//              ordered triggers.
// Neither h~(f) nor z(t) is written to memory.
#include "mf_filter.cuh"
#include "mf_sort.cuh"

namespace mf {

// ---------------------------------------------------------------------------
// per-unit set-up
// ---------------------------------------------------------------------------
// Unit i of a segment is template order[i] (bank order when order is NULL).
__global__ void k_units(SegDev seg, const double *__restrict__ tmpl, int n_t, double f_low, float thr,
                        int log2D, const int *__restrict__ order, UnitInfo *__restrict__ units, FilterCtl *clear,
                        int *zero) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    chain_wait(i);
    if (clear && blockIdx.x == 0) clear_ctl(clear);
    if (zero && i == 0) *zero = 0;
    if (i >= n_t) return;
    const int t = order ? order[i] : i;
    units[i] = unit_info(seg, tmpl + (int64_t)t * kTmplStride, t, f_low, thr, log2D);
}

__global__ void k_anchors(SegDev seg, const double *__restrict__ tmpl, const UnitInfo *__restrict__ units,
                          int unit0, int log2D, int max_anc, float4 *__restrict__ anchors,
                          float *__restrict__ anchors4, int reps) {
    int b = blockIdx.y;
    chain_wait(b);
    const UnitInfo u = units[unit0 + b];
    unit_anchors(seg, tmpl + (int64_t)u.tmpl * kTmplStride, u, log2D, max_anc, anchors + (int64_t)b * max_anc,
                 anchors4 + (int64_t)b * max_anc, reps, (int64_t)gridDim.y * max_anc,   // copy k of slot b: slot b + k n_units
                 blockIdx.x, gridDim.x);
}

__global__ void k_anchors64(SegDev seg, const double *__restrict__ tmpl, const UnitInfo *__restrict__ units, int unit0,
                            int log2D, int max_anc, float4 *__restrict__ anchors) {
    int b = blockIdx.y;
    chain_wait(b);
    const UnitInfo u = units[unit0 + b];
    const double *T = tmpl + (int64_t)u.tmpl * kTmplStride;
    const double c1 = T[TF_C1], c2 = T[TF_C2], c3 = T[TF_C3], c5 = T[TF_C5];
    float4 *out = anchors + (int64_t)b * 3 * max_anc;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < u.n_anc; i += gridDim.x * blockDim.x) {
        const int64_t g = (int64_t)u.g_lo + i;
        const Anchor64 r = anchor_record64(c1, c2, c3, c5, g, log2D, seg.df);
        const int64_t a = anchor_slot_index(g, seg.log2N, seg.log2N1, log2D);
        if (!MF_DBG(a >= 0 && a < max_anc, kDbgAnchor)) continue;
        auto lo = [](unsigned long long x) { return __int_as_float((int)(unsigned)x); };
        auto hi = [](unsigned long long x) { return __int_as_float((int)(unsigned)(x >> 32)); };
        out[a] = make_float4(lo(r.r0), hi(r.r0), lo(r.q1), hi(r.q1));
        out[a + max_anc] = make_float4(lo(r.q2), hi(r.q2), lo(r.q3), hi(r.q3));
        out[a + 2 * (int64_t)max_anc] = make_float4(r.q4, r.q5, r.q6, r.q7);
    }
}

// turns[k], k < N/2: the phase that pass 1 of MF_PHASE_FP64 hands to its sincos
// (mf_debug_phase), from the same two functions; 0 outside the template's band
__global__ void k_phase64(SegDev seg, const double *__restrict__ tmpl, int t, double f_low, int log2D,
                          double *__restrict__ turns) {
    int64_t k0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    chain_wait(k0);
    const double *T = tmpl + (int64_t)t * kTmplStride;
    const UnitInfo u = unit_info(seg, T, t, f_low, 0.f, log2D);
    for (int64_t k = k0; k < seg.N / 2; k += (int64_t)gridDim.x * blockDim.x) {
        double out = 0.0;
        if (k >= u.k_lo && k < u.k_hi) {
            const int64_t g = k >> log2D;
            const Anchor64 r = anchor_record64(T[TF_C1], T[TF_C2], T[TF_C3], T[TF_C5], g, log2D, seg.df);
            auto lo = [](unsigned long long x) { return __int_as_float((int)(unsigned)x); };
            auto hi = [](unsigned long long x) { return __int_as_float((int)(unsigned)(x >> 32)); };
            const int d = (int)(k - ((g << log2D) + ((1 << log2D) >> 1)));
            const float df = (float)d;
            unsigned sign;
            out = (double)anchor_phase64(make_float4(lo(r.r0), hi(r.r0), lo(r.q1), hi(r.q1)),
                                         make_float4(lo(r.q2), hi(r.q2), lo(r.q3), hi(r.q3)),
                                         make_float4(r.q4, r.q5, r.q6, r.q7), d, df, (df * df) * (df * df), sign);
            if (sign) out += 0.5;
        }
        turns[k] = out;
    }
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
MF_DEBUG_READER(dbg_read_filter)

cudaError_t launch_units(const SegDev &seg, const double *tmpl, int n_t, double f_low, float thr, int log2D,
                         const int *order, UnitInfo *units, FilterCtl *clear, cudaStream_t st, int *zero) {
    return launch(k_units, dim3((n_t + 255) / 256), 256, 0, st, seg, tmpl, n_t, f_low, thr, log2D, order, units, clear,
                  zero);
}

cudaError_t launch_anchors(const SegDev &seg, const double *tmpl, const UnitInfo *units, int unit0, int n_units,
                           int log2D, int max_anc, float4 *anchors, float *anchors4, int phase_mode, cudaStream_t st,
                           int reps) {
    if (reps < 1) return cudaErrorInvalidValue;
    const int per = 256;
    int gx = (max_anc + per - 1) / per;
    if (gx > 64) gx = 64;
    if (phase_mode == MF_PHASE_FP64) {
        if (reps != 1) return cudaErrorInvalidValue;
        return launch(k_anchors64, dim3(gx, n_units), per, 0, st, seg, tmpl, units, unit0, log2D, max_anc, anchors);
    }
    return launch(k_anchors, dim3(gx, n_units), per, 0, st, seg, tmpl, units, unit0, log2D, max_anc, anchors, anchors4,
                  reps);
}

cudaError_t launch_phase64(const SegDev &seg, const double *tmpl, int t, double f_low, int log2D, double *turns,
                           cudaStream_t st) {
    return launch(k_phase64, dim3((unsigned)((seg.N / 2 + 255) / 256)), 256, 0, st, seg, tmpl, t, f_low, log2D, turns);
}

namespace {
struct Pass1Op {
    const SegDev &seg;
    const UnitInfo *units;
    int unit0, n_units, log2D, max_anc, phase_mode;
    const float4 *anchors;
    const float *anchors4;
    float2 *exch;
    const double *tmpl;
    int anc_slots;
    bool narrow;
    cudaStream_t st;
    template <int N2, int N1>
    cudaError_t run() {
        constexpr int C = seqs_per_cta<N2>(N1);
        typename ExchSink<N2, C, +1, cx_ilog2(N1)>::Params kp{exch, seg.log2N1, seg.log2N};
        const dim3 grid(N1 / C, n_units);
        if (phase_mode == MF_PHASE_FP32) {
            typename TemplateSrcF32<N2, C, cx_ilog2(N1)>::Params sp{seg.W, units, tmpl, (float)seg.df};
            return run_pass<N2, C, true, +1, TemplateSrcF32<N2, C, cx_ilog2(N1)>, ExchSink<N2, C, +1, cx_ilog2(N1)>>(grid, sp, kp, st, unit0);
        }
        if (phase_mode == MF_PHASE_FP64) {
            typename TemplateSrc64<N2, C, cx_ilog2(N1)>::Params sp{seg.W, units, anchors, max_anc, log2D, anc_slots};
            return run_pass<N2, C, true, +1, TemplateSrc64<N2, C, cx_ilog2(N1)>, ExchSink<N2, C, +1, cx_ilog2(N1)>>(grid, sp, kp, st, unit0);
        }
        typename TemplateSrc<N2, C, cx_ilog2(N1)>::Params sp{seg.W, units, anchors, anchors4, max_anc, log2D, anc_slots};
        if (narrow)
            return run_pass<N2, C, true, +1, TemplateSrcNarrow<N2, C, cx_ilog2(N1)>, ExchSink<N2, C, +1, cx_ilog2(N1)>>(grid, sp, kp, st, unit0);
        return run_pass<N2, C, true, +1, TemplateSrc<N2, C, cx_ilog2(N1)>, ExchSink<N2, C, +1, cx_ilog2(N1)>>(grid, sp, kp, st, unit0);
    }
};

struct Pass2Op {
    const SegDev &seg;
    const UnitInfo *units;
    int unit0, n_units;
    const float2 *exch;
    float4 *partials;
    int seg_idx;
    KeyLayout kl;
    mf_trigger *staged;
    uint64_t *keys;
    unsigned long long *counter;
    int64_t cap;
    cudaStream_t st;
    template <int N2, int N1>
    cudaError_t run() {
        constexpr int C = seqs_per_cta<N1>(N2);
        const int nblk = N2 / C;
        typename RowSrc<N1, C>::Params sp{exch, seg.log2N1, seg.log2N};
        typename RhoSink<N1, C>::Params kp{units, partials, staged, keys, counter, cap,
                                           seg.log2N2, nblk, seg_idx, kl};
        return run_pass<N1, C, false, +1, RowSrc<N1, C>, RhoSink<N1, C>>(dim3(nblk, n_units), sp, kp, st, unit0);
    }
};

struct BlocksOp {
    int nblk = 0;
    template <int N2, int N1>
    cudaError_t run() {
        nblk = N2 / seqs_per_cta<N1>(N2);
        return cudaSuccess;
    }
};

struct AttrOp {
    template <int N2, int N1>
    cudaError_t run() {
        constexpr int C1 = seqs_per_cta<N2>(N1);
        constexpr int C2 = seqs_per_cta<N1>(N2);
        cudaError_t e;
        if ((e = set_pass_attrs<N2, C1, true, +1, TemplateSrc<N2, C1, cx_ilog2(N1)>, ExchSink<N2, C1, +1, cx_ilog2(N1)>>())) return e;
        if ((e = set_pass_attrs<N2, C1, true, +1, TemplateSrcNarrow<N2, C1, cx_ilog2(N1)>, ExchSink<N2, C1, +1, cx_ilog2(N1)>>())) return e;
        if ((e = set_pass_attrs<N2, C1, true, +1, TemplateSrcF32<N2, C1, cx_ilog2(N1)>, ExchSink<N2, C1, +1, cx_ilog2(N1)>>())) return e;
        if ((e = set_pass_attrs<N2, C1, true, +1, TemplateSrc64<N2, C1, cx_ilog2(N1)>, ExchSink<N2, C1, +1, cx_ilog2(N1)>>())) return e;
        return set_pass_attrs<N1, C2, false, +1, RowSrc<N1, C2>, RhoSink<N1, C2>>();
    }
};
}  // namespace

cudaError_t launch_pass1(const SegDev &seg, const UnitInfo *units, int unit0, int n_units, int log2D, int max_anc,
                         const float4 *anchors, const float *anchors4, float2 *exch, int phase_mode,
                         const double *tmpl, int p1_form, int *status, long long spin_limit, cudaStream_t st,
                         int form, int anc_slots) {
    if (p1_form != 1 && pass1_pf_applies(seg.log2N, seg.log2N2, log2D, phase_mode))
        return launch_pass1_pf(seg, units, unit0, n_units, log2D, max_anc, anchors, anchors4, exch, p1_form == 2,
                               status, spin_limit, st, form);
    Pass1Op op{seg, units, unit0, n_units, log2D, max_anc, phase_mode, anchors, anchors4, exch, tmpl, anc_slots, form == kBandNarrow, st};
    return dispatch_split2(seg.log2N, seg.log2N2, op);
}

cudaError_t launch_pass2(const SegDev &seg, const UnitInfo *units, int unit0, int n_units, const float2 *exch,
                         float4 *partials, int seg_idx, KeyLayout kl, mf_trigger *staged, uint64_t *keys,
                         unsigned long long *counter, int64_t cap, cudaStream_t st) {
    Pass2Op op{seg, units, unit0, n_units, exch, partials, seg_idx, kl, staged, keys, counter, cap, st};
    return dispatch_split2(seg.log2N, seg.log2N2, op);
}

int pass2_blocks(int log2N, int log2N2) {
    BlocksOp op;
    dispatch_split2(log2N, log2N2, op);
    return op.nblk;
}

cudaError_t filter_kernel_attributes() {
    {
        cudaError_t e0 = init_pass_tables();
        if (e0 != cudaSuccess) return e0;
    }
    for (int lg = 10; lg <= 22; ++lg) {
        AttrOp op;
        cudaError_t e = dispatch_split(lg, op);
        if (e == cudaSuccess && alt_log2n2(lg) > 0) e = dispatch_split2(lg, alt_log2n2(lg), op);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// peaks: one warp per unit reduces the pass-2 partials of that unit
// ---------------------------------------------------------------------------
__global__ void k_reduce_peaks(const UnitInfo *__restrict__ units, int n_units, const float4 *__restrict__ partials,
                               int nblk, int seg_idx, int n_seg, mf_peak *__restrict__ peaks) {
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    chain_wait(warp);
    if (warp >= n_units) return;
    unit_peak(units[warp], n_units, partials + (int64_t)warp * nblk, nblk, seg_idx, n_seg, peaks);
}

cudaError_t launch_reduce_peaks(const SegDev &seg, const UnitInfo *units, int n_units, const float4 *partials,
                                int nblk, int seg_idx, int n_seg, mf_peak *peaks, cudaStream_t st) {
    (void)seg;
    const int threads = 256;
    const int blocks = (n_units * 32 + threads - 1) / threads;
    return launch(k_reduce_peaks, dim3(blocks), threads, 0, st, units, n_units, partials, nblk, seg_idx, n_seg, peaks);
}

// ---------------------------------------------------------------------------
// Trigger compaction: the staged records into the caller's buffer in (tmpl,
// seg, j) order, by a stable LSD radix sort of the packed keys with 8-bit
// digits or, up to 16384 triggers, by rank (mf_sort.cuh), in one launch.
// ---------------------------------------------------------------------------
constexpr size_t kRankSmem = (size_t)kRankChunk * sizeof(uint64_t) + kSortThreads * sizeof(uint32_t);
constexpr size_t kTriggerSortSmem = sizeof(SortShared) > kRankSmem ? sizeof(SortShared) : kRankSmem;
__global__ void __launch_bounds__(kSortThreads, 1)
    k_sort_triggers(const unsigned long long *counter, int64_t cap, int key_bits, const mf_trigger *staged, uint64_t *keys, uint64_t *keys_tmp, uint32_t *idx_a,
                    uint32_t *idx_b, SortCtl *ctl, uint64_t *tstat, mf_trigger *__restrict__ out,
                    int64_t *__restrict__ n_out, int *status, int64_t spin_limit) {
    __shared__ __align__(16) unsigned char sort_smem[kTriggerSortSmem];
    SortShared &sh = *reinterpret_cast<SortShared *>(sort_smem);
    chain_wait(counter, staged);
    const unsigned long long total = *counter;
    const int64_t n = (int64_t)(total < (unsigned long long)cap ? total : (unsigned long long)cap);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *n_out = (int64_t)total;
        if (total > (unsigned long long)cap) atomicOr(status, 1);
    }
    if (n <= kRankMax && n <= (int64_t)gridDim.x * kSortThreads) {
        if (key_bits <= 32) sort_rank<uint32_t>(keys, (int)n, staged, out, sort_smem);
        else sort_rank<uint64_t>(keys, (int)n, staged, out, sort_smem);
        return;
    }
    const int npass = (key_bits + 7) / 8;
    const int64_t n_tiles = (n + kSortTile - 1) / kSortTile;
    if (!run_phase(ctl, 0, n_tiles, 0, sh, status, spin_limit, [&](int64_t t) {
            sort_hist_tile(ctl, tstat, t, n, npass, sh, [&](int64_t i) { return keys[i]; });
            return true;
        }))
        return;
    for (int p = 0; p < npass; ++p) {
        const uint64_t *kin = p & 1 ? keys_tmp : keys;
        const uint32_t *iin = p == 0 ? nullptr : (p & 1 ? idx_a : idx_b);
        if (!run_phase(ctl, 1 + p, n_tiles, n_tiles, sh, status, spin_limit, [&](int64_t t) {
                return sort_pass_tile(ctl, tstat, t, n, p, p == npass - 1, kin, iin, p & 1 ? keys : keys_tmp,
                                      p & 1 ? idx_b : idx_a, sh, spin_limit);
            }))
            return;
    }
    const uint32_t *perm = npass & 1 ? idx_a : idx_b;
    run_phase(ctl, 1 + npass, n_tiles, n_tiles, sh, status, spin_limit, [&](int64_t t) {
        gather_records(staged, out, t * kSortTile, min(n, (t + 1) * kSortTile), [&](int64_t i) { return __ldcg(&perm[i]); });
        return true;
    });
}

cudaError_t launch_sort_triggers(const unsigned long long *counter, int64_t cap, int key_bits,
                                 const mf_trigger *staged, const uint64_t *keys, uint64_t *keys_tmp,
                                 uint32_t *idx_a, uint32_t *idx_b, SortCtl *ctl, uint64_t *tstat, mf_trigger *out,
                                 int64_t *n_out, int *status, int n_sm, int64_t spin_limit, cudaStream_t st) {
    if (key_bits > 8 * kSortMaxPass) return cudaErrorInvalidValue;
    return launch(k_sort_triggers, dim3(n_sm), kSortThreads, 0, st, counter, cap, key_bits, staged,
                  const_cast<uint64_t *>(keys), keys_tmp, idx_a, idx_b, ctl, tstat, out, n_out, status, spin_limit);
}

}  // namespace mf
