// mf_sort.cuh -- stable LSD radix sort of 64-bit keys and the phase engine that
// runs a chain of dependent device-wide steps inside one launch.
//
// A search step ends with a sort of a few thousand trigger keys, and every
// kernel of a chain of small ones costs its launch (about 5 us of host time and
// a gap of 2 us on the device) more than its work: the sort of 5000 keys took a
// memset and 5 launches, 45 us.  So
//   sort_rank    up to 16384 unique keys: every CTA counts, for its share of the
//                keys, the smaller ones among all of them, which is their place:
//                no passes and no CTA waits for another;
//   sort_pass    more keys: tiles of 4096 keys with decoupled look-back (Merrill
//                & Garland's single-pass scan) per digit;
//   sort_small   up to 8192 keys inside one CTA (clustering), keys and payloads in
//                registers between passes and in shared memory for the scatter;
//   run_phase    hands the tiles of one step to the CTAs by a ticket counter and
//                lets a step's first tile of each CTA wait until every tile of
//                the step before is done.
// A CTA only ever waits for tiles that running CTAs hold (smaller tickets of the
// same step, or the step before), so the chain progresses whatever number of
// CTAs is resident; every wait is bounded all the same.
#pragma once
#include "mf_internal.h"

namespace mf {

constexpr int kSortThreads = 1024, kSortWarps = kSortThreads / 32;
constexpr int kSortSmallRows = 8, kSortSmall = kSortThreads * kSortSmallRows;   // one-CTA limit
constexpr int kSortRows = kSortTile / kSortThreads;

struct SortShared {
    uint32_t whist[kSortWarps][256];
    uint32_t base[256];
    uint32_t wsum[kSortWarps];
    int tile, ok;
};
// shared memory of a kernel with the one-CTA sort: SortShared, then its keys and payloads
constexpr size_t kSortSmemBytes = sizeof(SortShared) + (size_t)kSortSmall * (sizeof(uint64_t) + sizeof(uint32_t));
static_assert(sizeof(SortShared) % 8 == 0, "the keys follow the shared block");

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint64_t tstat_load(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void tstat_store(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Block-wide (all threads call it): true once *done >= target; false when the
// bound runs out or another CTA gave up.
__device__ __forceinline__ bool phase_wait(SortCtl *ctl, int phase, unsigned target, SortShared &sh, int *status,
                                           int64_t spin_limit) {
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t spins = 0;
        int ok = 1;
        while (ld_acquire(&ctl->done[phase]) < target) {
            if (ld_acquire(&ctl->abort) || ++spins > spin_limit) {
                atomicOr(status, 2);
                atomicExch(&ctl->abort, 1u);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        sh.ok = ok;
    }
    __syncthreads();
    return sh.ok != 0;
}

// Runs f(tile) for tiles of step `phase` (n_tiles of them) handed out by ticket;
// `before` tiles of step phase - 1 must be done first.  f returns false to give
// up.  All threads of the CTA call it.
template <class F>
__device__ __forceinline__ bool run_phase(SortCtl *ctl, int phase, int64_t n_tiles, int64_t before, SortShared &sh,
                                          int *status, int64_t spin_limit, F f) {
    bool waited = phase == 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) sh.tile = (int)atomicAdd(&ctl->ticket[phase], 1u);
        __syncthreads();
        const int64_t t = sh.tile;
        if (t >= n_tiles) return true;
        if (!waited) {
            if (!phase_wait(ctl, phase - 1, (unsigned)before, sh, status, spin_limit)) return false;
            waited = true;
        }
        if (!f(t)) {   // block-uniform
            if (threadIdx.x == 0) {
                atomicOr(status, 2);
                atomicExch(&ctl->abort, 1u);
            }
            return false;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&ctl->done[phase], 1u);
        }
    }
}

// exclusive prefix over 256 values, one per thread of the first 8 warps (all
// threads call it; the result is defined for threads < 256)
__device__ __forceinline__ uint32_t excl_scan_256(uint32_t x, SortShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh.wsum[warp] = incl;
    __syncthreads();
    uint32_t wo = 0;
    for (int w = 0; w < min(warp, 8); ++w) wo += sh.wsum[w];
    __syncthreads();
    return wo + incl - x;
}

// Lanes whose 8-bit digit equals this lane's, among the lanes with a digit
// (d < 256): one vote per bit (__match_any_sync takes as long: 28 us for 4400
// keys in one CTA either way).
__device__ __forceinline__ unsigned match_digit(uint32_t d) {
    unsigned peers = __ballot_sync(0xffffffffu, d < 256u);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned v = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        peers &= ((d >> b) & 1u) ? v : ~v;
    }
    return peers;
}

// Ranks rows of keys held by the warps (warp w owns ROWS rows of 32 consecutive
// keys, rows in order): lr[r] = the key's rank among the warp's equal digits,
// sh.whist[w][d] = the warp's count of digit d.  Inactive keys carry a digit
// >= 256.
template <int ROWS>
__device__ __forceinline__ void sort_rank_rows(const uint32_t *dg, uint32_t *lr, int rows, SortShared &sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    for (int e = lane; e < 256; e += 32) sh.whist[warp][e] = 0u;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r >= rows) break;
        const unsigned peers = match_digit(dg[r]);
        const uint32_t rank = (uint32_t)__popc(peers & lt_mask);
        const bool act = dg[r] < 256u;
        lr[r] = act ? sh.whist[warp][dg[r]] + rank : 0u;
        __syncwarp();
        if (act && rank == 0) sh.whist[warp][dg[r]] += (uint32_t)__popc(peers);
        __syncwarp();
    }
}

// whist[w][d] becomes the offset of warp w among digit d's keys of the tile;
// returns digit threadIdx.x's total (threads < 256)
__device__ __forceinline__ uint32_t sort_warp_offsets(SortShared &sh) {
    uint32_t tot = 0;
    if (threadIdx.x < 256) {
#pragma unroll 8
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = sh.whist[w][threadIdx.x];
            sh.whist[w][threadIdx.x] = tot;
            tot += c;
        }
    }
    return tot;
}

// One-CTA sort of n <= kSortSmall keys: key_of(i) gives key i; sidx[pos] = i at
// the end.  skey, sidx: shared memory of kSortSmall entries (key_of may read
// skey: all keys are loaded first).
template <class KeyOf>
__device__ __forceinline__ void sort_small(int n, int npass, SortShared &sh, uint64_t *skey, uint32_t *sidx,
                                           KeyOf key_of) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = (n + kSortThreads - 1) / kSortThreads;   // keys spread evenly: fewer rows per warp
    const int row0 = warp * 32 * rows + lane;
    uint64_t key[kSortSmallRows];
    uint32_t id[kSortSmallRows];
#pragma unroll
    for (int r = 0; r < kSortSmallRows; ++r) {
        const int i = row0 + r * 32;
        id[r] = (uint32_t)i;
        key[r] = (r < rows && i < n) ? key_of(i) : 0ull;
    }
    for (int p = 0; p < npass; ++p) {
        uint32_t dg[kSortSmallRows], lr[kSortSmallRows];
#pragma unroll
        for (int r = 0; r < kSortSmallRows; ++r)
            dg[r] = (r < rows && row0 + r * 32 < n) ? (uint32_t)(key[r] >> (8 * p)) & 255u : 256u + (uint32_t)lane;
        sort_rank_rows<kSortSmallRows>(dg, lr, rows, sh);
        __syncthreads();   // counts of every warp; every key of the last pass has been read back
        const uint32_t tot = sort_warp_offsets(sh);
        const uint32_t pre = excl_scan_256(tot, sh);
        if (threadIdx.x < 256) sh.base[threadIdx.x] = pre;
        __syncthreads();
        const bool last = p == npass - 1;
#pragma unroll
        for (int r = 0; r < kSortSmallRows; ++r) {
            if (dg[r] >= 256u) continue;
            const uint32_t pos = sh.base[dg[r]] + sh.whist[warp][dg[r]] + lr[r];
            sidx[pos] = id[r];
            if (!last) skey[pos] = key[r];
        }
        __syncthreads();
        if (!last) {
#pragma unroll
            for (int r = 0; r < kSortSmallRows; ++r) {
                const int i = row0 + r * 32;
                if (r < rows && i < n) {
                    key[r] = skey[i];
                    id[r] = sidx[i];
                }
            }
        }
    }
}

// Rank sort of n unique keys by all CTAs of the grid (kSortThreads threads
// each): CTA b places the records of keys [b k, b k + k), k = ceil(n / CTAs).
// Its threads are k keys times as many parts of the comparison as fit, so few
// keys are a few comparisons a thread and the latency of one read of the keys.
// The limit is where n^2 comparisons catch up with the radix passes: 4400 keys
// 28 us in one CTA's radix passes, 7 here, 180 keys 10 and 3.7; 22,800 keys 51 us
// in tiles and 75 here, so about 38 at the limit.
constexpr int kRankMax = 16384, kRankChunk = 4096;
template <class K>
__device__ __forceinline__ void sort_rank(const uint64_t *keys, int n, const mf_trigger *src, mf_trigger *dst,
                                          unsigned char *smem) {
    K *sk = reinterpret_cast<K *>(smem);
    uint32_t *rank = reinterpret_cast<uint32_t *>(smem + kRankChunk * sizeof(uint64_t));   // [kSortThreads]
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    const int k0 = (int)blockIdx.x * per, mine = min(per, n - k0);
    if (mine <= 0) return;
    const int parts = kSortThreads / per;   // the caller has n <= CTAs kSortThreads, so per <= kSortThreads
    const int q = (int)threadIdx.x % per, part = (int)threadIdx.x / per;
    const bool act = q < mine && part < parts;
    const K my = act ? (K)keys[k0 + q] : (K)0;
    if ((int)threadIdx.x < per) rank[threadIdx.x] = 0u;
    uint32_t less = 0;
    for (int c0 = 0; c0 < n; c0 += kRankChunk) {
        const int m = min(kRankChunk, n - c0);
        __syncthreads();
        for (int i = threadIdx.x; i < m; i += kSortThreads) sk[i] = (K)keys[c0 + i];
        __syncthreads();
        const int len = ((m + parts - 1) / parts + 3) & ~3;
        const int lo = part * len, hi = min(m, lo + len);
        if (act) {
            int j = lo;
#pragma unroll 4
            for (; j + 4 <= hi; j += 4) {
#pragma unroll
                for (int e = 0; e < 4; ++e) less += sk[j + e] < my ? 1u : 0u;
            }
            for (; j < hi; ++j) less += sk[j] < my ? 1u : 0u;
        }
    }
    if (act && less) atomicAdd(&rank[q], less);
    __syncthreads();
    constexpr int W = sizeof(mf_trigger) / 4;
    const uint32_t *s = reinterpret_cast<const uint32_t *>(src) + (int64_t)k0 * W;
    uint32_t *d = reinterpret_cast<uint32_t *>(dst);
    for (int w = threadIdx.x; w < mine * W; w += kSortThreads) {
        const int r = w / W;
        if (MF_DBG(rank[r] < (uint32_t)n, kDbgSort)) d[(int64_t)rank[r] * W + (w - r * W)] = s[w];
    }
}

// Digit histograms of one tile for every pass (into ctl->ghist) and its
// look-back words cleared.  key_of(i) gives key i < n.
template <class KeyOf>
__device__ __forceinline__ void sort_hist_tile(SortCtl *ctl, uint64_t *tstat, int64_t tile, int64_t n, int npass,
                                               SortShared &sh, KeyOf key_of) {
    for (int e = threadIdx.x; e < 256; e += kSortThreads) tstat[tile * 256 + e] = 0ull;
    uint32_t *h = &sh.whist[0][0];   // [pass][256]
    for (int e = threadIdx.x; e < npass * 256; e += kSortThreads) h[e] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
        const int64_t i = tile * kSortTile + r * kSortThreads + threadIdx.x;
        if (i < n) {
            const uint64_t k = key_of(i);
            for (int p = 0; p < npass; ++p) atomicAdd(&h[p * 256 + ((k >> (8 * p)) & 255u)], 1u);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < npass * 256; e += kSortThreads)
        if (h[e]) atomicAdd(&ctl->ghist[e], h[e]);
}

// dst[i] = src[index(i)] for i in [i0, i1), word by word with consecutive threads
// on consecutive words: whole-record copies by one thread each touch a sector
// per lane and word.  All threads call it.
template <class Index>
__device__ __forceinline__ void gather_records(const mf_trigger *src, mf_trigger *dst, int64_t i0, int64_t i1,
                                               Index index) {
    constexpr int W = sizeof(mf_trigger) / 4;
    const uint32_t *s = reinterpret_cast<const uint32_t *>(src);
    uint32_t *d = reinterpret_cast<uint32_t *>(dst) + i0 * W;
    const uint32_t n = (uint32_t)(i1 - i0) * W;
#pragma unroll 8
    for (uint32_t w = threadIdx.x; w < n; w += kSortThreads) {
        const uint32_t r = w / W;
        d[w] = __ldcg(&s[(int64_t)index(i0 + r) * W + (w - r * W)]);
    }
}

// One tile of one digit pass.  status word of (tile, digit) in tstat: bits
// 63..60 = pass + 1, bit 59 = inclusive prefix, bit 58 = tile aggregate, bits
// 31..0 = count.  The last pass writes the permutation iout only.  False when
// the bounded look-back gave up (block-uniform).
__device__ __forceinline__ bool sort_pass_tile(SortCtl *ctl, uint64_t *tstat, int64_t tile, int64_t n, int pass,
                                               bool last, const uint64_t *kin, const uint32_t *iin, uint64_t *kout,
                                               uint32_t *iout, SortShared &sh, int64_t spin_limit) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d_own = threadIdx.x;
    const uint64_t tag = (uint64_t)(pass + 1) << 60;
    const uint64_t kPrefix = 1ull << 59, kAgg = 1ull << 58;
    if (threadIdx.x == 0) sh.ok = 1;
    const uint32_t gpre = excl_scan_256(d_own < 256 ? __ldcg(&ctl->ghist[pass * 256 + d_own]) : 0u, sh);
    const int64_t row0 = tile * kSortTile + (int64_t)warp * (32 * kSortRows) + lane;
    uint64_t key[kSortRows];
    uint32_t id[kSortRows], dg[kSortRows], lr[kSortRows];
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
        const int64_t i = row0 + r * 32;
        const bool act = i < n;
        key[r] = act ? __ldcg(&kin[i]) : 0ull;
        id[r] = act ? (iin ? __ldcg(&iin[i]) : (uint32_t)i) : 0u;
        dg[r] = act ? (uint32_t)((key[r] >> (8 * pass)) & 255u) : (256u + (uint32_t)lane);
    }
    sort_rank_rows<kSortRows>(dg, lr, kSortRows, sh);
    __syncthreads();
    const uint32_t tot = sort_warp_offsets(sh);
    if (d_own < 256) {
        uint64_t *my = tstat + tile * 256 + d_own;
        uint32_t excl = 0;
        if (tile == 0) {
            tstat_store(my, tag | kPrefix | tot);
        } else {
            tstat_store(my, tag | kAgg | tot);
            int64_t pt = tile - 1, spins = 0;
            while (pt >= 0) {
                const uint64_t v = tstat_load(tstat + pt * 256 + d_own);
                if ((v >> 60) == (uint64_t)(pass + 1) && (v & (kPrefix | kAgg))) {
                    excl += (uint32_t)v;
                    if (v & kPrefix) break;
                    --pt;
                    continue;
                }
                if (++spins > spin_limit || ((spins & 255) == 0 && ld_acquire(&ctl->abort))) {
                    *(volatile int *)&sh.ok = 0;
                    break;
                }
                __nanosleep(32);
            }
            tstat_store(my, tag | kPrefix | (uint32_t)(excl + tot));
        }
        sh.base[d_own] = gpre + excl;
    }
    __syncthreads();
    if (!sh.ok) return false;
#pragma unroll
    for (int r = 0; r < kSortRows; ++r) {
        if (dg[r] >= 256u) continue;
        const uint32_t pos = sh.base[dg[r]] + sh.whist[warp][dg[r]] + lr[r];
        if (!MF_DBG(pos < (uint64_t)n, kDbgSort)) continue;
        iout[pos] = id[r];
        if (!last) kout[pos] = key[r];
    }
    return true;
}

}  // namespace mf
