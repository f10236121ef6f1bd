// mf_chisq.cu -- the chi^2 consistency test of Eq. (5) (Sec. 1.2) as a full
// time series, the computation the paper moved to the GPU: the band of
// Eq. (1) is split into p sub-bands of equal sigma^2 share, each sub-band's
// z_l(t) comes from its own inverse FFT, and
//   chi^2(t) = (p / sigma^2) sum_l |z_l(t) - z(t)/p|^2
//            = rho_scale^2 (p sum_l |raw_l(t)|^2 - |raw(t)|^2)     (sum_l z_l = z),
// with raw the pass-2 output of the filter (rho = |raw| rho_scale).
// Sub-band l is b_l <= k < b_{l+1}: b_0 = k_lo, b_p = k_hi and, for 0 < l < p,
// b_l is the smallest k with P[k] - P[k_lo] >= (l/p)(P[k_hi] - P[k_lo]), P the
// segment's FP64 prefix of f^(-7/3)/S (|h~|^2/S up to the amplitude).
// Each sub-band runs through the filter's own pass 1 (template generation on
// the sub-band only, column IFFTs) into its own exchange; one kernel then runs
// the row IFFTs of all p + 1 bands, summing |raw_l|^2 in registers and turning
// the sum into chi^2 at the full band.  Neither z_l nor z is stored.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "mf_filter.cuh"

namespace mf {

// One block per chi^2 unit: the sub-band edges by binary search in P, then
// p + 1 copies of the unit's full-band UnitInfo (band l = [b_l, b_{l+1}),
// band p = the full band).  A template index outside the bank gives an empty
// band (the output row is zero).
__global__ void k_chisq_units(SegDev seg, const UnitInfo *__restrict__ all, int n_t, const int32_t *__restrict__ tmpl,
                              int n, int p, UnitInfo *__restrict__ out, int64_t *__restrict__ edges) {
    __shared__ int64_t b[kChisqMaxBands + 1];
    int u = blockIdx.x;
    chain_wait(u);
    const int t = tmpl[u];
    UnitInfo full;
    if (t >= 0 && t < n_t) {
        full = all[t];
    } else {   // empty band on template 0's record (keeps every later read in range)
        full = all[0];
        full.k_hi = full.k_lo;
    }
    const int64_t lo = full.k_lo, hi = full.k_hi;
    const double P0 = seg.P[lo], Q = seg.P[hi] - P0;
    const int lane = threadIdx.x & 31;
    for (int l = threadIdx.x >> 5; l <= p; l += blockDim.x >> 5) {   // one warp per edge, 32 probes a step
        int64_t a = l == p ? hi : lo;
        if (l > 0 && l < p) {
            const double target = ((double)l / (double)p) * Q;
            a = edge_search(seg.P, P0, target, lo, hi, lane);
        }
        if (lane == 0) {
            b[l] = a;
            if (edges) edges[(int64_t)u * (p + 1) + l] = a;
        }
    }
    __syncthreads();
    for (int l = threadIdx.x; l <= p; l += blockDim.x) {
        UnitInfo x = full;
        if (l < p) {
            x.k_lo = (int32_t)b[l];
            x.k_hi = (int32_t)b[l + 1];
        }
        out[(int64_t)l * n + u] = x;
    }
}

// ---------------------------------------------------------------------------
// chi^2 tile kernel (row lengths other than 1024).  Pass 1 has written the
// exchange of every sub-band l = 0..p of a batch of nb templates, sub-band l
// of entry b at exch + (l nb + b) N.  Each CTA owns C rows j2 = tile C ..
// tile C + C - 1 of one entry and transforms them for l = 0..p in turn,
// summing |raw_l|^2 of its 32 outputs per thread in registers; at l = p (the
// full band) the sum becomes chi^2 = rho_scale^2 (p sum_l |raw_l|^2 - |raw|^2).
// The C consecutive samples of each j1 then leave through a shared-memory
// tile (per-element stores from the butterflies would touch one 32-byte sector
// per lane).  One launch per batch instead of one per sub-band, and no
// accumulator in memory: 16 templates at N = 2^16, p = 16 took 17 pass-1 and
// 17 pass-2 launches of 7 us each, every one a fraction of a wave: 330 us a
// call, 105 us now.
// ---------------------------------------------------------------------------
struct ChiTilesParams {
    float2 *exch;           // group sums are kept over bands already read
    const UnitInfo *full;   // full-band units of the call's template list
    float *chisq;           // [n][N]
    int unit0, nb, p;
    int log2N, log2N1, log2N2;
};

// rows of one sub-band; from the second sub-band on, the sequences' shared
// memory is free only once every thread has read its last stage
template <int L, int C, class Sync>
struct ChiTileSrc {
    static constexpr bool kHalfZero = false;
    const RowSrc<L, C> rows;
    const bool again;
    __device__ __forceinline__ void load(int seq, int t, float2 *v) const {
        rows.load(seq, t, v);
        if (again) Sync::sync();
    }
};
struct ChiWarpSync {
    static __device__ __forceinline__ void sync() { __syncwarp(); }
};

// p |raw_l|^2 of the thread's 32 outputs summed over the bands l < p it has seen
// since the last start, less |raw|^2 of the full band l = p.  The bands are taken
// in descending order, the one pass 1 wrote last first: of an exchange somewhat
// larger than L2 the ascending order finds nothing left.
struct ChiTileAcc {
    float acc[32];
    int l = 0, p = 0;
    float pf = 0.f;
    __device__ __forceinline__ void start() {
#pragma unroll
        for (int r = 0; r < 32; ++r) acc[r] = 0.f;
    }
    template <int R>
    __device__ __forceinline__ void store(int, int, int, const float2 *v) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float pw = fmaf(v[r].x, v[r].x, v[r].y * v[r].y);
            acc[r] = l == p ? -pw : fmaf(pf, pw, acc[r]);
        }
    }
    // kept in 16 float2 of this thread, T apart
    template <int T>
    __device__ __forceinline__ void put(float2 *x) const {
#pragma unroll
        for (int i = 0; i < 16; ++i) __stcg(&x[i * T], make_float2(acc[2 * i], acc[2 * i + 1]));
    }
    template <int T>
    __device__ __forceinline__ void add(const float2 *x) {   // acc = x + acc
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float2 v = __ldcg(&x[i * T]);
            acc[2 * i] = v.x + acc[2 * i];
            acc[2 * i + 1] = v.y + acc[2 * i + 1];
        }
    }
};

// Rows of up to 512 points: a sample's sum has one order whatever CTAs form it, so
// a template's chi^2 has the same bits alone and in every list.  The bands form
// four groups from p = 7 on, two from p = 3 on, each summed in descending order;
// the sum is (G3 + G2) + (G1 + G0) or G1 + G0.
template <int L>
__host__ __device__ constexpr bool chi_ordered() { return L <= 512; }
__host__ __device__ __forceinline__ int chi_groups(int p) { return p >= 7 ? 4 : (p >= 3 ? 2 : 1); }
__device__ __forceinline__ int chi_start(int g, int of, int p) { return (g * (p + 1) + of - 1) / of; }

// S > 1: a cluster of S CTAs shares a tile, CTA c taking the groups of part c of
// S; the CTAs add their sums through distributed shared memory, 1 / S of the tile
// each.  A CTA with several groups keeps the sums of all but its last where it
// has just read the band that begins the group: each warp over its own 1024
// points of the exchange, which nothing reads again.  A sum kept is 64 KB a tile
// more to move, 1 % of a call (200 templates at 2^16, p = 16: 881 us in one sum,
// 902 in four; pairs keep one each, 16 templates 103.7 -> 105.2; fours none, 9
// templates 89 -> 86).  Kept in 32 KB of shared memory the L1 that is left cannot
// hold the loads in flight (72 us for the 50 below), 32 more registers a thread
// would spill, and one sum in order over four CTAs, the lower ones adding their
// bands late, was 94 -> 105 us for 30 templates at 2^14.
// A tile a CTA leaves the GPU to a few: 16 templates at N = 2^16, p = 16, are 128
// tiles, 17 transforms of 3.6 us one after the other, 61 us; 50 us in pairs of CTAs
// whose warps (with their own rows) do not wait for one another: 59 with CTA
// barriers, 53 in ascending order.
template <int L, int C, int S>
__global__ void __launch_bounds__(C *(L / 32), (C * (L / 32) >= 256) ? 2 : 1) k_chisq_tiles(ChiTilesParams q) {
    extern __shared__ float2 chi_smem[];
    constexpr int T = L / 32, NT = C * T;
    static_assert(chi_ordered<L>() || S == 1, "clusters keep the order of the sum");
    // rows of up to 1024 points lie within a warp: no barrier holds the warps together
    using Sync = std::conditional_t<(L <= 1024), ChiWarpSync, CtaSync>;
    float2 *tw = chi_smem + pass_data_bytes<L, C>() / sizeof(float2);
    int tile = blockIdx.x / S, b = blockIdx.y;
    const int c = S > 1 ? (int)(blockIdx.x % S) : 0;   // rank in the cluster
    fill_twiddles<L>(tw);
    chain_wait(tile, b);
    const int groups = chi_ordered<L>() ? chi_groups(q.p) : 1;
    const int l0 = chi_start(c, S, q.p), l1 = chi_start(c + 1, S, q.p);
    // the bands that begin the groups 1, 2 (or the upper of two) and 3; a CTA's last group ends with l0
    const int b1 = groups == 4 ? chi_start(1, 4, q.p) : -1, b3 = groups == 4 ? chi_start(3, 4, q.p) : -1;
    const int b2 = groups > 1 ? chi_start(1, 2, q.p) : -1;
    const float rs = q.full[q.unit0 + b].rho_scale, rs2 = rs * rs;
    ChiTileAcc snk;
    snk.p = q.p;
    snk.pf = (float)q.p;
    snk.start();
    const int seq = threadIdx.x / T, t = threadIdx.x % T;
    auto kept = [&](int l) {   // over the 1024 points of the warp's rows, 256 bytes at a time
        return q.exch + ((int64_t)(l * q.nb + b) << q.log2N) + tile * C * L + ((int)threadIdx.x & ~31) * 32 + (threadIdx.x & 31);
    };
    const typename RowSrc<L, C>::Params rp{q.exch, q.log2N1, q.log2N};
    __syncthreads();   // twiddles
#pragma unroll 1
    for (int l = l1 - 1; l >= l0; --l) {
        snk.l = l;
        ChiTileSrc<L, C, Sync> src{RowSrc<L, C>(rp, tile, 0, l * q.nb + b, nullptr), l < l1 - 1};
        cta_fft<L, C, false, +1, ChiTileSrc<L, C, Sync>, ChiTileAcc, Sync>(chi_smem, tw, src, snk);
        if (chi_ordered<L>() && S < 4 && l > l0 && (l == b1 || l == b2 || l == b3)) {
            if (S == 1 && groups == 4 && l == b2) {   // G3 + G2, in the place of G3
                snk.template add<32>(kept(b3));
                snk.template put<32>(kept(b3));
            } else {
                snk.template put<32>(kept(l));
            }
            snk.start();
        }
    }
    if (chi_ordered<L>() && S < 4) {
        if (groups == 4) snk.template add<32>(kept(c > 0 ? b3 : b1));
        if (S == 1 && groups > 1) snk.template add<32>(kept(groups == 4 ? b3 : b2));
    }
    auto row = [&](int s) { return reinterpret_cast<float *>(chi_smem + s * SeqStride<L, C>::value); };
    __syncthreads();   // the last stage has read the sequences
    float *out = q.chisq + ((int64_t)(q.unit0 + b) << q.log2N) + tile * C;
    const float scale = S == 1 ? rs2 : 1.f;
#pragma unroll
    for (int r = 0; r < 32; ++r) row(seq)[t + r * T] = scale * snk.acc[r];
    if constexpr (S == 1) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < C * L; idx += NT) {
            const int s = idx % C, j1 = idx / C;
            __stcs(&out[s + ((int64_t)j1 << q.log2N2)], row(s)[j1]);
        }
    } else {
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        const float2 *peer[S];
#pragma unroll
        for (int i = 0; i < S; ++i) peer[i] = cl.map_shared_rank(chi_smem, i);
        cl.sync();
        for (int idx = c * (C * L / S) + threadIdx.x; idx < (c + 1) * (C * L / S); idx += NT) {
            const int s = idx % C, j1 = idx / C;
            auto sum = [&](int i) { return reinterpret_cast<const float *>(peer[i] + s * SeqStride<L, C>::value)[j1]; };
            float a = sum(1) + sum(0);
            if constexpr (S == 4) a = (sum(3) + sum(2)) + a;
            __stcs(&out[s + ((int64_t)j1 << q.log2N2)], rs2 * a);
        }
        cl.sync();   // no CTA leaves while its sums are being read
    }
}

// One band of one template (little memory: no p + 1 exchanges), l = p .. 0 in turn:
// the sums stay in sums[3][N] between the launches, the group's own, G3 (+ G2) or
// the upper of two, and G1.  The order of the sum is k_chisq_tiles'.
template <int L, int C>
__global__ void __launch_bounds__(C *(L / 32), (C * (L / 32) >= 256) ? 2 : 1)
    k_chisq_step(ChiTilesParams q, int l, float2 *sums) {
    extern __shared__ float2 chi_smem[];
    constexpr int T = L / 32, NT = C * T;
    using Sync = std::conditional_t<(L <= 1024), ChiWarpSync, CtaSync>;
    float2 *tw = chi_smem + pass_data_bytes<L, C>() / sizeof(float2);
    int tile = blockIdx.x;
    fill_twiddles<L>(tw);
    chain_wait(tile);
    const int groups = chi_ordered<L>() ? chi_groups(q.p) : 1;
    const int b1 = groups == 4 ? chi_start(1, 4, q.p) : -1, b3 = groups == 4 ? chi_start(3, 4, q.p) : -1;
    const int b2 = groups > 1 ? chi_start(1, 2, q.p) : -1;
    const float rs = q.full[q.unit0].rho_scale, rs2 = rs * rs;
    const int64_t half_n = (int64_t)1 << (q.log2N - 1);   // float2 of one of the sums
    float2 *own = sums + (int64_t)tile * (C * L / 2) + threadIdx.x, *hi = own + half_n, *lo = hi + half_n;
    ChiTileAcc snk;
    snk.l = l;
    snk.p = q.p;
    snk.pf = (float)q.p;
    snk.start();
    if (l < q.p && l + 1 != b1 && l + 1 != b2 && l + 1 != b3) snk.template add<NT>(own);   // 0 + x
    const typename RowSrc<L, C>::Params rp{q.exch, q.log2N1, q.log2N};
    __syncthreads();   // twiddles
    ChiTileSrc<L, C, Sync> src{RowSrc<L, C>(rp, tile, 0, 0, nullptr), false};
    cta_fft<L, C, false, +1, ChiTileSrc<L, C, Sync>, ChiTileAcc, Sync>(chi_smem, tw, src, snk);
    if (l > 0) {
        if (groups == 4 && l == b2) snk.template add<NT>(hi);
        snk.template put<NT>(l == b1 ? lo : (l == b2 || l == b3 ? hi : own));
        return;
    }
    if (groups == 4) snk.template add<NT>(lo);
    if (groups > 1) snk.template add<NT>(hi);
    const int seq = threadIdx.x / T, t = threadIdx.x % T;
    auto row = [&](int s) { return reinterpret_cast<float *>(chi_smem + s * SeqStride<L, C>::value); };
    __syncthreads();   // the last stage has read the sequences
#pragma unroll
    for (int r = 0; r < 32; ++r) row(seq)[t + r * T] = rs2 * snk.acc[r];
    __syncthreads();
    float *out = q.chisq + ((int64_t)q.unit0 << q.log2N) + tile * C;
    for (int idx = threadIdx.x; idx < C * L; idx += NT) {
        const int s = idx % C, j1 = idx / C;
        __stcs(&out[s + ((int64_t)j1 << q.log2N2)], row(s)[j1]);
    }
}

// ---------------------------------------------------------------------------
// chi^2 rows kernel (N1 = 1024, N = 2^19 and 2^20).  Pass 1 has written the
// exchange of every sub-band l = 0..p of a batch of nb templates, sub-band l
// of entry b at exch + (l nb + b) N.  Each warp owns one row j2 of one entry
// and transforms it for l = 0..p in turn: the row arrives by a bulk copy
// (cp.async.bulk, mbarrier, bounded wait), stage 0 runs from the staged row,
// and once the last stage has read the warp's region the copy of the same row
// of sub-band l + 1 is issued, so it lands under the arithmetic.  |raw_l|^2 is
// summed in registers over l < p and |raw|^2 (l = p) kept, so
//   chi^2 = rho_scale^2 (p sum_l |raw_l|^2 - |raw|^2)
// is formed without any accumulator in memory.  The CTA's 8 warps own 8
// consecutive rows; they park their 1024 values each in their regions and
// write the 8 x 1024 tile with 8 consecutive samples per 32-byte sector.
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ uint32_t cs_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cs_mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cs_addr(bar)) : "memory");
}
__device__ __forceinline__ bool cs_mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(cs_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// generic-proxy accesses of this thread before the async-proxy refill of its region
__device__ __forceinline__ void cs_fence_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cs_row_copy(float2 *dst, const float2 *src, uint64_t *bar) {
    constexpr uint32_t bytes = 1024 * sizeof(float2);
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                     cs_addr(bar)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     cs_addr(dst)),
                 "l"(src), "r"(bytes), "r"(cs_addr(bar))
                 : "memory");
}

constexpr int kChiWarps = 8;

struct ChiRowsParams {
    const float2 *exch;
    const UnitInfo *full;   // full-band units of the call's template list
    float *chisq;           // [n][N]
    int unit0, nb, p;
    int log2N, log2N2;
    int *status;            // bit 2: a wait ran out
    long long spin_limit;
    int stall;              // test hook: the row copies of list entry `stall` are never issued (-1: none)
};

// last-stage sink: |raw_l|^2 of the thread's 32 outputs (t + 32 q) summed over
// l < p; at l = p (the full band) the sum becomes chi^2 in place; refills the
// region with the next sub-band's row
struct ChiRowAcc {
    float acc[32];
    int l = 0, p = 0;
    float pf = 0.f, rs2 = 0.f;
    float2 *region = nullptr;
    uint64_t *bar = nullptr;
    const float2 *next_src = nullptr;
    __device__ __forceinline__ void after_loads() {
        __syncwarp();
        cs_fence_proxy();
        if (next_src != nullptr && (threadIdx.x & 31) == 0) cs_row_copy(region, next_src, bar);
    }
    template <int R>
    __device__ __forceinline__ void store(int, int, int, const float2 *v) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float pw = fmaf(v[r].x, v[r].x, v[r].y * v[r].y);
            if (l < p) acc[r] = l == 0 ? pw : acc[r] + pw;
            else acc[r] = rs2 * fmaf(pf, acc[r], -pw);
        }
    }
};

__device__ __forceinline__ bool chi_withheld(const ChiRowsParams &p, int64_t r) {
    return p.unit0 + (int)(r >> p.log2N2) == p.stall;
}

__device__ __forceinline__ const float2 *chi_row_src(const ChiRowsParams &p, int64_t r, int l) {
    const int64_t b = r >> p.log2N2, j2 = r & (((int64_t)1 << p.log2N2) - 1);
    if (!MF_DBG(b < p.nb && l <= p.p && ((j2 + 1) << 10) <= ((int64_t)1 << p.log2N), kDbgRows)) return p.exch;
    return p.exch + (((int64_t)l * p.nb + b) << p.log2N) + (j2 << 10);
}

__global__ void __launch_bounds__(kChiWarps * 32, 2) k_chisq_rows(ChiRowsParams p) {
    constexpr int L = 1024;
    using S = FftShape<L>;
    extern __shared__ __align__(16) float2 chi_rows_smem[];
    float2 *tw = chi_rows_smem + kChiWarps * S::STRIDE;
    uint64_t *bars = reinterpret_cast<uint64_t *>(tw + TwTable<L>::SIZE);
    const int w = threadIdx.x >> 5, t = threadIdx.x & 31;
    float2 *region = chi_rows_smem + w * S::STRIDE;
    fill_twiddles<L>(tw);
    if (t == 0) cs_mbar_init(&bars[w]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    int64_t r0 = (int64_t)blockIdx.x * kChiWarps;
    chain_wait_async(r0);
    // rows of the batch: nb N2, a multiple of 8 (N2 >= 512), so every warp has a row in every round
    const int64_t total = (int64_t)p.nb << p.log2N2;
    const int64_t step = (int64_t)gridDim.x * kChiWarps;
    const float pf = (float)p.p;
    if (r0 < total && t == 0 && !chi_withheld(p, r0 + w)) cs_row_copy(region, chi_row_src(p, r0 + w, 0), &bars[w]);
    uint32_t parity = 0;
    // a warp whose wait ran out stops waiting and issues no further copies
    // (none of its copies is then in flight), but keeps to the CTA barriers
    bool dead = false;
    for (; r0 < total; r0 += step) {
        const int64_t r = r0 + w;
        ChiRowAcc snk;
        snk.p = p.p;
        snk.pf = pf;
        {
            const float rs = p.full[p.unit0 + (int)(r >> p.log2N2)].rho_scale;
            snk.rs2 = rs * rs;
        }
        snk.region = region;
        snk.bar = &bars[w];
        for (int l = 0; l <= p.p; ++l) {
            // the row of sub-band l has landed (bounded; on expiry the warp is
            // marked dead and the status bit set at the end)
            if (!dead) {
                long long it = 0;
                bool got = true;
                while (!cs_mbar_try_wait(&bars[w], parity)) {
                    if (++it > p.spin_limit) { got = false; break; }
                }
                dead = !__all_sync(0xffffffffu, got);
                parity ^= 1u;
            }
            float2 v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = region[t + 32 * q];
            Dft<32, +1>::run(v);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 32; ++q) region[spad(32 * t + q)] = v[q];
            __syncwarp();
            snk.l = l;
            // the next row's first copy waits for the flush
            snk.next_src = (l < p.p && !dead && !chi_withheld(p, r)) ? chi_row_src(p, r, l + 1) : nullptr;
            stockham_stage<L, S::R1, 32, +1, true, ChiRowAcc, ChiWarpSync>(region, tw, 0, t, snk);
        }
        // chi^2 of the row's 1024 samples j2 + N2 (t + 32 q), parked in the warp's region
        float *rowf = reinterpret_cast<float *>(region);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 32; ++q) rowf[t + 32 * q] = snk.acc[q];
        __syncthreads();
        // the CTA's 8 rows j2 .. j2 + 7 of entry b: 8 consecutive samples per j1
        const int64_t jb = r0 & (((int64_t)1 << p.log2N2) - 1);
        float *out = p.chisq + ((int64_t)(p.unit0 + (r0 >> p.log2N2)) << p.log2N) + jb;
        for (int idx = threadIdx.x; idx < kChiWarps * L; idx += kChiWarps * 32) {
            const int s = idx & (kChiWarps - 1), j1 = idx >> 3;
            __stcs(&out[s + ((int64_t)j1 << p.log2N2)],
                   reinterpret_cast<const float *>(chi_rows_smem + s * S::STRIDE)[j1]);
        }
        cs_fence_proxy();
        __syncthreads();   // the tile is read: the regions may be refilled
        const int64_t rn = r + step;
        if (rn < total && t == 0 && !dead && !chi_withheld(p, rn)) cs_row_copy(region, chi_row_src(p, rn, 0), &bars[w]);
    }
    if (dead && t == 0 && p.status != nullptr) atomicOr(p.status, 2);
}

static size_t chi_rows_smem_bytes() {
    return (size_t)kChiWarps * FftShape<1024>::STRIDE * sizeof(float2) + (size_t)TwTable<1024>::SIZE * sizeof(float2) +
           kChiWarps * sizeof(uint64_t);
}

template <int L, int C>
constexpr size_t chi_tiles_smem_bytes() {
    return pass_data_bytes<L, C>() + (size_t)TwTable<L>::SIZE * sizeof(float2);
}

struct ChiTilesOp {
    const ChiTilesParams *q;   // NULL: set the kernel attributes only
    int n_sm;
    cudaStream_t st;
    int step = -1;             // >= 0: this band alone, with sums
    float2 *sums = nullptr;
    template <int N2, int N1, int S>
    cudaError_t tiles() {
        constexpr int C = seqs_per_cta<N1>(N2);
        constexpr size_t smem = chi_tiles_smem_bytes<N1, C>();
        if (!q)
            return cudaFuncSetAttribute(k_chisq_tiles<N1, C, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return launch_in_clusters(k_chisq_tiles<N1, C, S>, dim3(S * (N2 / C), q->nb), C * (N1 / 32), S > 1 ? S : 0, smem, st, *q);
    }
    template <int N2, int N1>
    cudaError_t run() {
        if constexpr (N1 != 1024) {
            constexpr int C = seqs_per_cta<N1>(N2);
            constexpr size_t smem = chi_tiles_smem_bytes<N1, C>();
            if (q && step >= 0)
                return launch(k_chisq_step<N1, C>, dim3(N2 / C), C * (N1 / 32), smem, st, *q, step, sums);
            if (!q) {
                cudaError_t e = cudaFuncSetAttribute(k_chisq_step<N1, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return e;
            }
            if constexpr (chi_ordered<N1>()) {   // a template of 2048-point rows is 256 tiles and more
                if (!q) {
                    cudaError_t e = tiles<N2, N1, 2>();
                    if (e == cudaSuccess) e = tiles<N2, N1, 4>();
                    if (e != cudaSuccess) return e;
                } else {
                    // as many CTAs per tile as keep the launch within one wave (two per
                    // SM), with a group each, of two sub-bands or more
                    const int64_t n = (int64_t)(N2 / C) * q->nb, wave = 2 * (int64_t)n_sm;
                    if (4 * n <= wave && chi_groups(q->p) == 4) return tiles<N2, N1, 4>();
                    if (2 * n <= wave && chi_groups(q->p) >= 2) return tiles<N2, N1, 2>();
                }
            }
            return tiles<N2, N1, 1>();
        } else {
            return q ? cudaErrorInvalidValue : cudaSuccess;   // 1024-point rows: k_chisq_rows
        }
    }
};
}  // namespace

cudaError_t launch_chisq_units(const SegDev &seg, const UnitInfo *all, int n_t, const int32_t *tmpl, int n, int p,
                               UnitInfo *out, int64_t *edges, cudaStream_t st) {
    if (p < 1 || p > kChisqMaxBands) return cudaErrorInvalidValue;
    return launch(k_chisq_units, dim3(n), p >= 8 ? 256 : 128, 0, st, seg, all, n_t, tmpl, n, p, out, edges);
}

cudaError_t launch_chisq_tiles(const SegDev &seg, float2 *exch, const UnitInfo *full, int unit0, int nb, int p,
                               float *chisq, int n_sm, cudaStream_t st) {
    ChiTilesParams q{exch, full, chisq, unit0, nb, p, seg.log2N, seg.log2N1, seg.log2N2};
    ChiTilesOp op{&q, n_sm, st};
    return dispatch_split(seg.log2N, op);
}

bool chisq_rows_applies(int log2N) { return log2N - log2_n2(log2N) == 10; }

cudaError_t launch_chisq_step(const SegDev &seg, float2 *exch, const UnitInfo *full, int unit, int l, int p, float2 *sums,
                              float *chisq, cudaStream_t st) {
    ChiTilesParams q{exch, full, chisq, unit, 1, p, seg.log2N, seg.log2N1, seg.log2N2};
    ChiTilesOp op{&q, 0, st, l, sums};
    return dispatch_split(seg.log2N, op);
}

cudaError_t launch_chisq_rows(const SegDev &seg, const float2 *exch, const UnitInfo *full, int unit0, int nb, int p,
                              float *chisq, int *status, long long spin_limit, int stall, int n_sm, cudaStream_t st) {
    if (!chisq_rows_applies(seg.log2N) || nb < 1) return cudaErrorInvalidValue;
    ChiRowsParams q{exch, full, chisq, unit0, nb, p, seg.log2N, seg.log2N2, status, spin_limit, stall};
    const int64_t rounds = ((int64_t)nb << seg.log2N2) / kChiWarps;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(2 * (int64_t)n_sm, rounds));
    return launch(k_chisq_rows, dim3(grid), kChiWarps * 32, chi_rows_smem_bytes(), st, q);
}

MF_DEBUG_READER(dbg_read_chisq)

cudaError_t chisq_kernel_attributes() {
    {
        cudaError_t e0 = init_twiddle_tables();
        if (e0 != cudaSuccess) return e0;
    }
    {
        cudaError_t e1 = cudaFuncSetAttribute(k_chisq_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)chi_rows_smem_bytes());
        if (e1 != cudaSuccess) return e1;
    }
    for (int lg = 10; lg <= 22; ++lg) {
        ChiTilesOp op{nullptr, 0, nullptr};
        cudaError_t e = dispatch_split(lg, op);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace mf
