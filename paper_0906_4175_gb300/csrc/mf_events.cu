// mf_events.cu -- events from triggers, and the chi^2 of Eq. (5) at single
// samples.
//
// Clustering (the paper reports events, Sec. 3.3, and gives no rule): single
// linkage in time with a maximum gap of `window` samples, first over the
// triggers of each (template, segment) pair (input sorted by (tmpl, seg, j)),
// then over those clusters' loudest members of all templates within a
// segment (re-sorted by (seg, j, tmpl)).  A cluster's representative is its
// loudest member, the earliest in the pass's order on ties.  Each pass is
//   start flags -> inclusive scan (cluster ids) -> packed atomicMax of
//   (rho bits, ~index) and member counts per cluster -> emit,
// all in one launch, with the record count read on the device, so the host
// never synchronises.
//
// chi^2 at a sample (Eq. 5 at t = j dt): the sub-band sums of Eq. (1),
//   R_l = sum_{k in [b_l, b_{l+1})} W_k e^{-i Psi_k} e^{2 pi i j k / N},
//   chi^2 = p (P_tot/Q) sum_l |R_l - R/p|^2,  R = sum_l R_l,
// with the sub-band edges of mf_chisq_series and the filter's phase form
// (FP64 anchors, FP32 quartic Taylor, FP32 sincos); (j k mod N) is exact in
// integers.  One row per point, blocks over the band, FP64 block totals per
// sub-band in a fixed order.
#include "mf_filter.cuh"
#include "mf_sort.cuh"
#include "mf_tmpl.cuh"

namespace mf {

// ---------------------------------------------------------------------------
// clustering: one launch.  Up to 8192 triggers one CTA does everything in shared
// memory; more go through the steps below as tiles (run_phase).  As twenty
// kernels (flags, three-kernel scans, reductions, a six-launch sort) 5000
// triggers took 105 us, launches and their gaps almost all of it.
// ---------------------------------------------------------------------------
struct ClusterParams {
    const mf_trigger *trig;
    const int64_t *n_trig;
    int64_t cap;
    int window, npass;
    KeyLayout kl;
    ClusterScratch w;
    mf_event *events;
    int64_t ev_cap;
    int64_t *n_events;
    int64_t spin_limit;
};

// record i of a pass starts a cluster (mode 1: per (tmpl, seg), mode 2: per seg)
__device__ __forceinline__ bool cl_starts(const mf_trigger &a, const mf_trigger &b, int window, int mode) {
    const bool same = mode == 1 ? (a.tmpl == b.tmpl && a.seg == b.seg) : (a.seg == b.seg);
    return !(same && (int64_t)b.j - (int64_t)a.j <= window);
}
// the same for record i = t of a warp's consecutive records; before(i) loads record i (lane 0's predecessor)
template <class Before>
__device__ __forceinline__ bool cl_lane_starts(const mf_trigger &t, int64_t i, int window, int mode, Before before) {
    mf_trigger a;
    a.tmpl = __shfl_up_sync(0xffffffffu, t.tmpl, 1);
    a.seg = __shfl_up_sync(0xffffffffu, t.seg, 1);
    a.j = __shfl_up_sync(0xffffffffu, t.j, 1);
    if (i == 0) return true;
    if ((threadIdx.x & 31) == 0) a = before(i - 1);
    return cl_starts(a, t, window, mode);
}
__device__ __forceinline__ unsigned long long cl_key(float rho, uint32_t i) {
    return ((unsigned long long)__float_as_uint(fmaxf(rho, 0.f)) << 32) | (0xffffffffull - (unsigned long long)i);
}
__device__ __forceinline__ uint32_t cl_index(unsigned long long best) {
    return (uint32_t)(0xffffffffull - (best & 0xffffffffull));
}
__device__ __forceinline__ uint64_t cl_sort_key(const mf_trigger &r, const KeyLayout &kl) {
    return ((uint64_t)r.seg << (kl.j_bits + kl.tmpl_bits)) | ((uint64_t)r.j << kl.tmpl_bits) | (uint64_t)r.tmpl;
}
__device__ __forceinline__ mf_event cl_event(const mf_trigger &r, uint32_t n_trig, uint32_t n_tmpl) {
    mf_event e;
    e.tmpl = r.tmpl;
    e.seg = r.seg;
    e.j = r.j;
    e.rho = r.rho;
    e.z_re = r.z_re;
    e.z_im = r.z_im;
    e.n_trig = (int32_t)n_trig;
    e.n_tmpl = (int32_t)n_tmpl;
    return e;
}

// Runs of equal cluster id c over the warp's lanes (ids do not decrease with
// the lane; c = 0xffffffff: inactive): the run's first lane gets the maximum of
// key and the sums of one and of weight, and true.
__device__ __forceinline__ bool cl_warp_run(uint32_t c, unsigned long long &key, uint32_t &count, uint32_t &weight) {
    const int lane = threadIdx.x & 31;
    count = 1u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t oc = __shfl_down_sync(0xffffffffu, c, o);
        const unsigned long long ok = __shfl_down_sync(0xffffffffu, key, o);
        const uint32_t on = __shfl_down_sync(0xffffffffu, count, o), ow = __shfl_down_sync(0xffffffffu, weight, o);
        if (lane + o < 32 && oc == c) {
            if (ok > key) key = ok;
            count += on;
            weight += ow;
        }
    }
    const uint32_t before = __shfl_up_sync(0xffffffffu, c, 1);
    return c != 0xffffffffu && (lane == 0 || before != c);
}

// Cluster ids of ROWS x 1024 records (record r * 1024 + threadIdx.x; flag bits
// in fl): local inclusive count of starts - 1 into id[], returns the total.
template <int ROWS>
__device__ __forceinline__ uint32_t cl_ids(uint32_t fl, uint32_t *id, SortShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *cnt = &sh.whist[0][0];   // [row][warp]: starts per warp, then their exclusive prefix
    static_assert(ROWS * kSortWarps <= 256, "one value per thread of the scan");
    uint32_t bal[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        bal[r] = __ballot_sync(0xffffffffu, (fl >> r) & 1u);
        if (lane == 0) cnt[r * kSortWarps + warp] = (uint32_t)__popc(bal[r]);
    }
    __syncthreads();
    const uint32_t x = threadIdx.x < ROWS * kSortWarps ? cnt[threadIdx.x] : 0u;
    const uint32_t ex = excl_scan_256(x, sh);
    if (threadIdx.x < ROWS * kSortWarps) cnt[threadIdx.x] = ex;
    if (threadIdx.x == ROWS * kSortWarps - 1) sh.base[0] = ex + x;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
        id[r] = cnt[r * kSortWarps + warp] + (uint32_t)__popc(bal[r] & (0xffffffffu >> (31 - lane))) - 1u;
    const uint32_t total = sh.base[0];
    __syncthreads();
    return total;
}

// One CTA, n <= kSortSmall records.
__device__ __forceinline__ void cluster_small(const ClusterParams &p, int n, unsigned char *smem) {
    SortShared &sh = *reinterpret_cast<SortShared *>(smem);
    uint64_t *skey = reinterpret_cast<uint64_t *>(smem + sizeof(SortShared));   // best of a cluster, then sort keys
    uint32_t *sidx = reinterpret_cast<uint32_t *>(skey + kSortSmall);
    uint32_t *rep = sidx + kSortSmall;       // trigger index of a pass-1 cluster's loudest member
    uint32_t *members = rep + kSortSmall;    // its trigger count
    unsigned long long *best = reinterpret_cast<unsigned long long *>(skey);
    uint32_t *sums = &sh.whist[0][0];        // pass 2: members << 16 | triggers (both <= 8192)
    constexpr int R = kSortSmallRows;
    const int tid = threadIdx.x;
    uint32_t id[R];
    // pass 1: per (template, segment); a record's predecessor is the previous
    // lane's, lane 0 loads it
    uint32_t fl = 0;
    float rho[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * kSortThreads + tid;
        best[i] = 0ull;
        members[i] = 0u;
        if (r * kSortThreads < n) {
            const mf_trigger t = p.trig[min(i, n - 1)];
            rho[r] = t.rho;
            if (cl_lane_starts(t, i, p.window, 1, [&](int64_t q) { return p.trig[min(q, (int64_t)n - 1)]; }) && i < n) fl |= 1u << r;
        }
    }
    const int nc = (int)cl_ids<R>(fl, id, sh);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * kSortThreads + tid;
        if (r * kSortThreads >= n) break;
        unsigned long long key = i < n ? cl_key(rho[r], (uint32_t)i) : 0ull;
        uint32_t count, weight = 0u;
        const uint32_t c = i < n ? id[r] : 0xffffffffu;
        if (cl_warp_run(c, key, count, weight)) {
            atomicMax(&best[c], key);
            atomicAdd(&members[c], count);
        }
    }
    __syncthreads();
    for (int c = tid; c < nc; c += kSortThreads) {
        const uint32_t i = cl_index(best[c]);
        rep[c] = i;
        skey[c] = cl_sort_key(p.trig[i], p.kl);
    }
    __syncthreads();
    // the representatives in (seg, j, tmpl) order: sidx[pos] = cluster
    sort_small(nc, p.npass, sh, skey, sidx, [&](int i) { return skey[i]; });
    // pass 2: across templates within a segment
    fl = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * kSortThreads + tid;
        if (r * kSortThreads < nc) {
            const mf_trigger t = p.trig[rep[sidx[min(i, nc - 1)]]];
            rho[r] = t.rho;
            if (cl_lane_starts(t, i, p.window, 2, [&](int64_t q) { return p.trig[rep[sidx[min(q, (int64_t)nc - 1)]]]; }) && i < nc) fl |= 1u << r;
        }
    }
    const int ne = (int)cl_ids<R>(fl, id, sh);
    for (int i = tid; i < kSortSmall; i += kSortThreads) {
        best[i] = 0ull;
        sums[i] = 0u;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * kSortThreads + tid;
        if (r * kSortThreads >= nc) break;
        unsigned long long key = i < nc ? cl_key(rho[r], (uint32_t)i) : 0ull;
        uint32_t count, weight = i < nc ? members[sidx[i]] : 0u;
        const uint32_t c = i < nc ? id[r] : 0xffffffffu;
        if (cl_warp_run(c, key, count, weight)) {
            atomicMax(&best[c], key);
            atomicAdd(&sums[c], (count << 16) | weight);
        }
    }
    __syncthreads();
    if (tid == 0) *p.n_events = ne;
    for (int c = tid; c < ne && c < p.ev_cap; c += kSortThreads) {
        const uint32_t w = sums[c];
        p.events[c] = cl_event(p.trig[rep[sidx[cl_index(best[c])]]], w & 0xffffu, w >> 16);
    }
}

// Start flags, cluster ids (look-back over the tiles' start counts: bit 63 =
// inclusive prefix, bit 62 = tile count, bits 31..0 the value) and the
// reductions of one tile of records; the last tile writes the cluster count.
__device__ __forceinline__ bool cl_scan_tile(const ClusterParams &p, const mf_trigger *rec, int64_t n, int64_t tile,
                                             int64_t n_tiles, int mode, uint64_t *scan, unsigned long long *best,
                                             uint32_t *members, uint32_t *wsum, const uint32_t *perm, int64_t *n_out,
                                             SortShared &sh) {
    constexpr int R = kSortRows;
    uint32_t id[R], fl = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = tile * kSortTile + r * kSortThreads + threadIdx.x;
        if (i < n && (i == 0 || cl_starts(rec[i - 1], rec[i], p.window, mode))) fl |= 1u << r;
    }
    if (threadIdx.x == 0) sh.ok = 1;
    const uint32_t total = cl_ids<R>(fl, id, sh);
    if (threadIdx.x == 0) {
        uint32_t excl = 0;
        if (tile > 0) {
            tstat_store(&scan[tile], (1ull << 62) | total);
            int64_t pt = tile - 1, spins = 0;
            while (pt >= 0) {
                const uint64_t v = tstat_load(&scan[pt]);
                if (v >> 62) {
                    excl += (uint32_t)v;
                    if (v >> 63) break;
                    --pt;
                    continue;
                }
                if (++spins > p.spin_limit || ((spins & 255) == 0 && ld_acquire(&p.w.ctl->abort))) {
                    sh.ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        tstat_store(&scan[tile], (1ull << 63) | (uint32_t)(excl + total));
        sh.base[1] = excl;
        if (tile == n_tiles - 1) *n_out = (int64_t)excl + total;
    }
    __syncthreads();
    if (!sh.ok) return false;
    const uint32_t excl = sh.base[1];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t i = tile * kSortTile + r * kSortThreads + threadIdx.x;
        const bool act = i < n;
        unsigned long long key = act ? cl_key(rec[i].rho, (uint32_t)i) : 0ull;
        uint32_t count, weight = act && wsum ? __ldcg(&p.w.members[__ldcg(&perm[i])]) : 0u;
        const uint32_t c = act ? excl + id[r] : 0xffffffffu;
        if (cl_warp_run(c, key, count, weight)) {
            atomicMax(&best[c], key);
            atomicAdd(&members[c], count);
            if (wsum) atomicAdd(&wsum[c], weight);
        }
    }
    return true;
}

// The steps of a call of more than kSortSmall records, as tiles.  A CTA whose
// wait runs out sets ctl->abort and returns.
__device__ __forceinline__ void cluster_tiles(const ClusterParams &p, int64_t n, unsigned char *smem) {
    SortShared &sh = *reinterpret_cast<SortShared *>(smem);
    const ClusterScratch &w = p.w;
    const int64_t tn = (n + kSortTile - 1) / kSortTile;
    auto items = [&](int64_t t, int64_t count, auto f) {
        for (int r = 0; r < kSortRows; ++r) {
            const int64_t i = t * kSortTile + r * kSortThreads + threadIdx.x;
            if (i < count) f(i);
        }
        return true;
    };
    int ph = 0;
    // accumulators and look-back words
    if (!run_phase(w.ctl, ph, tn, 0, sh, w.status, p.spin_limit, [&](int64_t t) {
            if (threadIdx.x < 2) w.scan[2 * t + threadIdx.x] = 0ull;
            return items(t, n, [&](int64_t i) {
                w.best[i] = w.best2[i] = 0ull;
                w.members[i] = w.members2[i] = w.wsum[i] = 0u;
            });
        }))
        return;
    // pass 1: per (template, segment)
    uint64_t *scan1 = w.scan, *scan2 = w.scan + tn;
    ++ph;
    if (!run_phase(w.ctl, ph, tn, tn, sh, w.status, p.spin_limit, [&](int64_t t) {
            return cl_scan_tile(p, p.trig, n, t, tn, 1, scan1, w.best, w.members, nullptr, nullptr, w.n_c, sh);
        }))
        return;
    if (!phase_wait(w.ctl, ph, (unsigned)tn, sh, w.status, p.spin_limit)) return;
    const int64_t nc = __ldcg(w.n_c), tc = (nc + kSortTile - 1) / kSortTile;
    // representatives, their sort keys and digit histograms
    ++ph;
    if (!run_phase(w.ctl, ph, tc, tn, sh, w.status, p.spin_limit, [&](int64_t t) {
            items(t, nc, [&](int64_t c) {
                const mf_trigger r = p.trig[cl_index(__ldcg(&w.best[c]))];
                w.rep[c] = r;
                w.keys[c] = cl_sort_key(r, p.kl);
            });
            sort_hist_tile(w.ctl, w.tstat, t, nc, p.npass, sh, [&](int64_t i) { return w.keys[i]; });   // own writes
            return true;
        }))
        return;
    for (int q = 0; q < p.npass; ++q) {
        ++ph;
        const uint64_t *kin = q & 1 ? w.keys_tmp : w.keys;
        const uint32_t *iin = q == 0 ? nullptr : (q & 1 ? w.idx_a : w.idx_b);
        if (!run_phase(w.ctl, ph, tc, tc, sh, w.status, p.spin_limit, [&](int64_t t) {
                return sort_pass_tile(w.ctl, w.tstat, t, nc, q, q == p.npass - 1, kin, iin, q & 1 ? w.keys : w.keys_tmp,
                                      q & 1 ? w.idx_b : w.idx_a, sh, p.spin_limit);
            }))
            return;
    }
    const uint32_t *perm = p.npass & 1 ? w.idx_a : w.idx_b;
    ++ph;
    if (!run_phase(w.ctl, ph, tc, tc, sh, w.status, p.spin_limit, [&](int64_t t) {
            gather_records(w.rep, w.sorted, t * kSortTile, min(nc, (t + 1) * kSortTile),
                           [&](int64_t i) { return __ldcg(&perm[i]); });
            return true;
        }))
        return;
    // pass 2: across templates within a segment
    ++ph;
    if (!run_phase(w.ctl, ph, tc, tc, sh, w.status, p.spin_limit, [&](int64_t t) {
            return cl_scan_tile(p, w.sorted, nc, t, tc, 2, scan2, w.best2, w.members2, w.wsum, perm, w.n_c + 1, sh);
        }))
        return;
    if (!phase_wait(w.ctl, ph, (unsigned)tc, sh, w.status, p.spin_limit)) return;
    const int64_t ne = __ldcg(w.n_c + 1), m = ne < p.ev_cap ? ne : p.ev_cap;
    ++ph;
    run_phase(w.ctl, ph, (m + kSortTile - 1) / kSortTile, tc, sh, w.status, p.spin_limit, [&](int64_t t) {
        return items(t, m, [&](int64_t c) {
            p.events[c] = cl_event(w.sorted[cl_index(__ldcg(&w.best2[c]))], __ldcg(&w.wsum[c]), __ldcg(&w.members2[c]));
        });
    });
}

__global__ void __launch_bounds__(kSortThreads, 1) k_cluster(const __grid_constant__ ClusterParams p) {
    extern __shared__ __align__(16) unsigned char cl_smem[];
    const int64_t nt = *p.n_trig;
    const int64_t n = nt < p.cap ? (nt > 0 ? nt : 0) : p.cap;
    if (n <= kSortSmall) {
        if (blockIdx.x == 0) {
            if (n == 0) {
                if (threadIdx.x == 0) *p.n_events = 0;
            } else {
                cluster_small(p, (int)n, cl_smem);
            }
        }
        return;
    }
    cluster_tiles(p, n, cl_smem);
    // The last CTA to leave writes the count, or -1 where any of them gave up:
    // the caller sees that there is no result, whatever stage it was lost in.
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&p.w.ctl->left, 1u) == gridDim.x - 1) {
            __threadfence();
            *p.n_events = ld_acquire(&p.w.ctl->abort) ? -1 : __ldcg(p.w.n_c + 1);
        }
    }
}

constexpr size_t kClusterSmem = kSortSmemBytes + 2 * (size_t)kSortSmall * sizeof(uint32_t);

cudaError_t launch_cluster(const mf_trigger *trig, const int64_t *n_trig, int64_t cap, int window, KeyLayout kl,
                           const ClusterScratch &w, mf_event *events, int64_t ev_cap, int64_t *n_events, int n_sm,
                           int64_t spin_limit, cudaStream_t st) {
    const int key_bits = kl.j_bits + kl.seg_bits + kl.tmpl_bits;
    const int npass = key_bits > 0 ? (key_bits + 7) / 8 : 1;
    if (npass > kSortMaxPass) return cudaErrorInvalidValue;
    ClusterParams p{trig, n_trig, cap, window, npass, kl, w, events, ev_cap, n_events, spin_limit};
    k_cluster<<<cap <= kSortSmall ? 1 : n_sm, kSortThreads, kClusterSmem, st>>>(p);
    return cudaGetLastError();
}

cudaError_t events_kernel_attributes() {
    return cudaFuncSetAttribute(k_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem);
}

// ---------------------------------------------------------------------------
// chi^2 at single samples
// ---------------------------------------------------------------------------
// Bound: latency.  A call has a few to a few hundred rows, each a sum over up to
// N/2 bins that 4..64 blocks share, so what a block does before and after its
// bins counts: the anchor spacing comes from the host (the bank's, as in the
// filter), the sub-band edges from a 32-way search by one warp per edge (4
// dependent loads instead of 20), sub-bands outside a block's bins cost
// nothing, and the row's total is one warp per sub-band instead of one thread
// per row.  9 rows at N = 2^20, p = 16: 85 + 175 us before, 36 + 7 us now.
constexpr int kCpThreads = 256, kCpWarps = kCpThreads / 32;
constexpr int kCpAnchors = kCpThreads;

template <int NS>
struct CpSegs {
    SegDev s[NS];
    int lg[NS];   // log2 of the anchor spacing (0: FP64 phase at every bin)
    int n;
};

struct CpRow {
    double c[4];
    int64_t b[kChisqMaxBands + 1];
    double pratio;
};

// band [k_lo, k_hi) of the row's template (empty for an invalid row) and P_tot / Q
__device__ __forceinline__ void cp_band(const SegDev &seg, double f_low, double fisco, bool valid, int64_t &lo,
                                        int64_t &hi, double &pratio) {
    const double N = (double)seg.N, fs = seg.fs;
    const double fc = fisco < 0.5 * fs ? fisco : 0.5 * fs;
    lo = (int64_t)ceil(f_low * N / fs);
    hi = (int64_t)floor(fc * N / fs) + 1;
    if (lo < 1) lo = 1;
    if (hi > seg.N / 2) hi = seg.N / 2;
    if (hi < lo || !valid) hi = lo;
    const double Q = seg.P[hi] - seg.P[lo];
    pratio = Q > 0.0 ? seg.consts->P_tot / Q : 0.0;
}

// interior sub-band edges (the rule and arithmetic of k_chisq_units: the
// smallest k with P[k] - P[lo] >= (l/p) Q) as far as they lie inside (r0, r1);
// the others are clamped to r0 or r1, which is all the caller needs.  One warp
// per edge, 32 probes a step.
__device__ void cp_row_edges(const SegDev &seg, int p, int64_t r0, int64_t r1, CpRow &r) {
    const int lane = threadIdx.x & 31;
    const int64_t lo = r.b[0], hi = r.b[p];
    const double P0 = seg.P[lo], Q = seg.P[hi] - P0, C0 = seg.P[r0] - P0, C1 = seg.P[r1] - P0;
    for (int l = 1 + (threadIdx.x >> 5); l < p; l += kCpWarps) {
        const double target = ((double)l / (double)p) * Q;
        int64_t a = r0;
        if (C1 < target) a = r1;
        else if (C0 < target) a = edge_search(seg.P, P0, target, r0, r1, lane);
        if (lane == 0) r.b[l] = a;
    }
}

__device__ __forceinline__ bool cp_row_valid(int32_t t, int n_t, int32_t sg, int n_seg, int32_t j, const SegDev &seg) {
    return t >= 0 && t < n_t && sg >= 0 && sg < n_seg && j >= 0 && (int64_t)j < seg.N;
}

// partial[(row * p + l) * bpr + block] = (re, im) of R_l over this block's bins
template <int NS>
__global__ void __launch_bounds__(kCpThreads)
    k_chisq_points(const __grid_constant__ CpSegs<NS> segs, const double *__restrict__ tmpl, int n_t, double f_low,
                   const int32_t *__restrict__ rows, int64_t stride, int p, double2 *__restrict__ partial,
                   double *__restrict__ pratio) {
    __shared__ CpRow row;
    __shared__ float4 sanc[kCpAnchors];
    __shared__ float sanc4[kCpAnchors];
    __shared__ double red[2][kCpWarps];
    int64_t i = blockIdx.y;
    chain_wait(i);
    const int32_t t = rows[i * stride], sg = rows[i * stride + 1], jj = rows[i * stride + 2];
    const int si = sg >= 0 && sg < segs.n ? sg : 0;
    const SegDev &seg = segs.s[si];
    const bool valid = cp_row_valid(t, n_t, sg, segs.n, jj, seg);
    if (threadIdx.x == 0) {
        const double *T = tmpl + (int64_t)(valid ? t : 0) * kTmplStride;
        row.c[0] = T[TF_C1]; row.c[1] = T[TF_C2]; row.c[2] = T[TF_C3]; row.c[3] = T[TF_C5];
        cp_band(seg, f_low, T[TF_FISCO], valid, row.b[0], row.b[p], row.pratio);
    }
    __syncthreads();
    const uint32_t nmask = (uint32_t)(seg.N - 1), j = (uint32_t)(valid ? jj : 0);
    const int64_t k_lo = row.b[0], k_hi = row.b[p];
    // this block's bin range: whole anchor groups (or a plain chunk in the FP64 form)
    const int log2D = segs.lg[si];
    const int lg = log2D > 0 ? log2D : 8;
    const int64_t g_lo = k_lo >> lg, g_hi = k_hi > k_lo ? ((k_hi - 1) >> lg) : g_lo - 1;
    const int64_t ng = g_hi - g_lo + 1;
    const int64_t gpb = (ng + gridDim.x - 1) / gridDim.x;
    const int64_t gb0 = g_lo + (int64_t)blockIdx.x * gpb;
    const int64_t gb1 = (gb0 + gpb < g_lo + ng) ? gb0 + gpb : g_lo + ng;
    int64_t r0 = gb0 << lg, r1 = gb1 << lg;
    if (r0 < k_lo) r0 = k_lo;
    if (r1 > k_hi) r1 = k_hi;
    if (r0 >= r1) {   // no bins for this block: zero sums
        for (int l = threadIdx.x; l < p; l += kCpThreads)
            partial[(i * p + l) * gridDim.x + blockIdx.x] = make_double2(0.0, 0.0);
        if (blockIdx.x == 0 && threadIdx.x == 0) pratio[i] = row.pratio;
        return;
    }
    cp_row_edges(seg, p, r0, r1, row);
    if (blockIdx.x == 0 && threadIdx.x == 0) pratio[i] = row.pratio;
    __syncthreads();
    const float invN = 1.0f / (float)seg.N;
    const int half = (1 << lg) >> 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double2 *out = partial + i * p * gridDim.x + blockIdx.x;
    for (int l = 0; l < p; ++l) {
        const int64_t a = row.b[l] > r0 ? row.b[l] : r0, b = row.b[l + 1] < r1 ? row.b[l + 1] : r1;
        if (a >= b) {   // no bin of this sub-band here (block-uniform)
            if (threadIdx.x == 0) out[(int64_t)l * gridDim.x] = make_double2(0.0, 0.0);
            continue;
        }
        float sr = 0.f, si_ = 0.f;
        // anchors of the groups this sub-band slice touches, in chunks of kCpAnchors
        for (int64_t k0 = a; k0 < b;) {
            const int64_t ga = k0 >> lg;
            int64_t ge = ga + kCpAnchors;
            int64_t kend = ge << lg;
            if (kend > b) kend = b;
            if (log2D > 0) {
                const int64_t gend = ((kend - 1) >> lg) + 1;
                if (ga + threadIdx.x < gend)
                    anchor_record(row.c[0], row.c[1], row.c[2], row.c[3], ga + threadIdx.x, lg, seg.df,
                                  sanc[threadIdx.x], sanc4[threadIdx.x]);
                __syncthreads();
            }
            for (int64_t k = k0 + threadIdx.x; k < kend; k += kCpThreads) {
                float psi;
                if (log2D > 0) {
                    const int ai = (int)((k >> lg) - ga);
                    const float4 an = sanc[ai];
                    const float d = (float)(int)((k & ((1 << lg) - 1)) - half);
                    psi = an.x + d * (an.y + d * (an.z + d * (an.w + d * sanc4[ai])));
                } else {
                    const double f = (double)k * seg.df;
                    double u = (double)rcbrtf((float)f);
                    u = u * (4.0 - f * u * u * u) * (1.0 / 3.0);
                    double ps = -0.125 + u * (row.c[0] + u * (row.c[1] + u * (row.c[2] + u * u * row.c[3])));
                    psi = (float)(ps - rint(ps));
                }
                float ph = (float)(((uint32_t)k * j) & nmask) * invN - psi;
                ph -= rintf(ph);
                float sn, cs;
                __sincosf(6.283185307179586f * ph, &sn, &cs);
                const float2 w = __ldg(&seg.W[k]);
                sr += w.x * cs - w.y * sn;
                si_ += w.x * sn + w.y * cs;
            }
            if (log2D > 0) __syncthreads();
            k0 = kend;
        }
        // block totals of this sub-band (FP64, fixed order)
        double vr = sr, vi = si_;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            vr += __shfl_xor_sync(0xffffffffu, vr, o);
            vi += __shfl_xor_sync(0xffffffffu, vi, o);
        }
        if (lane == 0) { red[0][warp] = vr; red[1][warp] = vi; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double tr = 0.0, ti = 0.0;
            for (int w = 0; w < kCpWarps; ++w) { tr += red[0][w]; ti += red[1][w]; }
            out[(int64_t)l * gridDim.x] = make_double2(tr, ti);
        }
        __syncthreads();
    }
}

// one CTA per row: a warp sums the blocks of a sub-band (fixed order), then one
// warp forms chi^2
template <int NS>
__global__ void __launch_bounds__(kCpThreads)
    k_chisq_points_final(const __grid_constant__ CpSegs<NS> segs, int n_t, const int32_t *__restrict__ rows,
                         int64_t stride, int p, const double2 *__restrict__ partial, const double *__restrict__ pratio,
                         int bpr, float *__restrict__ chisq) {
    __shared__ double2 R[kChisqMaxBands];
    int64_t i = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    chain_wait(i);
    const int32_t t = rows[i * stride], sg = rows[i * stride + 1], jj = rows[i * stride + 2];
    if (!cp_row_valid(t, n_t, sg, segs.n, jj, segs.s[sg >= 0 && sg < segs.n ? sg : 0])) {
        if (threadIdx.x == 0) chisq[i] = __int_as_float(0x7fc00000);
        return;
    }
    for (int l = warp; l < p; l += kCpWarps) {
        const double2 *q = partial + (i * p + l) * bpr;
        double vr = 0.0, vi = 0.0;
        for (int b = lane; b < bpr; b += 32) {
            const double2 v = q[b];
            vr += v.x;
            vi += v.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            vr += __shfl_xor_sync(0xffffffffu, vr, o);
            vi += __shfl_xor_sync(0xffffffffu, vi, o);
        }
        if (lane == 0) R[l] = make_double2(vr, vi);
    }
    __syncthreads();
    if (warp != 0) return;
    double Rr = 0.0, Ri = 0.0;
    for (int l = lane; l < p; l += 32) {
        Rr += R[l].x;
        Ri += R[l].y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Rr += __shfl_xor_sync(0xffffffffu, Rr, o);
        Ri += __shfl_xor_sync(0xffffffffu, Ri, o);
    }
    Rr /= p;
    Ri /= p;
    double s = 0.0;
    for (int l = lane; l < p; l += 32) {
        const double dr = R[l].x - Rr, di = R[l].y - Ri;
        s += dr * dr + di * di;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) chisq[i] = (float)((double)p * pratio[i] * s);
}

// The segment table travels as a kernel parameter: the smallest of three sizes
// that holds the call's segments (88 bytes each; 256 of them cost the launch).
template <int NS>
static cudaError_t chisq_points_run(const SegDev *segs, const int *lg, int n_seg, const double *tmpl, int n_t,
                                    double f_low, const int32_t *rows, int64_t stride, int64_t n, int p, int bpr,
                                    double2 *partial, double *pratio, float *chisq, cudaStream_t st) {
    CpSegs<NS> tab;
    for (int s = 0; s < n_seg; ++s) {
        tab.s[s] = segs[s];
        tab.lg[s] = lg[s];
    }
    tab.n = n_seg;
    const cudaError_t e = launch(k_chisq_points<NS>, dim3((unsigned)bpr, (unsigned)n), kCpThreads, 0, st, tab, tmpl, n_t,
                                 f_low, rows, stride, p, partial, pratio);
    if (e != cudaSuccess) return e;
    return launch(k_chisq_points_final<NS>, dim3((unsigned)n), kCpThreads, 0, st, tab, n_t, rows, stride, p, partial, pratio,
                  bpr, chisq);
}

cudaError_t launch_chisq_points(const SegDev *segs, const int *lg, int n_seg, const double *tmpl, int n_t,
                                double f_low, const int32_t *rows, int64_t stride, int64_t n, int p, int bpr,
                                double2 *partial, double *pratio, float *chisq, cudaStream_t st) {
    if (n_seg < 1 || n_seg > kRefineMaxSegs || p < 1 || p > kChisqMaxBands) return cudaErrorInvalidValue;
    auto run = n_seg == 1 ? chisq_points_run<1> : (n_seg <= 16 ? chisq_points_run<16> : chisq_points_run<kRefineMaxSegs>);
    return run(segs, lg, n_seg, tmpl, n_t, f_low, rows, stride, n, p, bpr, partial, pratio, chisq, st);
}

}  // namespace mf
