// mf_group.cu -- short segments of one filter call in common launches.
//
// A bank of a hundred templates over a segment of 2^10 .. 2^16 samples is a few
// dozen tiles of 8192 points: every kernel of the chain (units and anchors, pass
// 1, pass 2, peaks) is a part of one wave and takes its latency, not its work,
// and segment after segment 26 us at 75 templates; 4 segments of 2^12 .. 2^14 106 us, 62 together.  Up to kGroupMax such
// segments, of any mix of lengths, share each of the four launches: the blocks
// are dealt out over (segment, unit, tile) and a block takes the transform of
// its segment's length.  The tile code is that of the per-tile kernels, so
// every output bit is the same.
#include "mf_filter.cuh"

namespace mf {

namespace {
constexpr int kGroupThreads = 256;

// the segment whose blocks [end[s-1], end[s]) hold block b; b becomes its index there
__device__ __forceinline__ int group_find(const int *end, int n, int &b) {
    int s = 0;
    while (s + 1 < n && b >= end[s]) ++s;
    if (s > 0) b -= end[s - 1];
    return s;
}

template <int N2, int N1>
constexpr size_t group_smem() {
    constexpr int C1 = seqs_per_cta<N2>(N1), C2 = seqs_per_cta<N1>(N2);
    constexpr size_t a = pass_smem_bytes<N2, C1, TemplateSrc<N2, C1, cx_ilog2(N1)>>();
    constexpr size_t b = pass_smem_bytes<N1, C2, RowSrc<N1, C2>>();
    return a > b ? a : b;
}
constexpr size_t smax(size_t a, size_t b) { return a > b ? a : b; }
constexpr size_t kGroupSmem =
    smax(smax(smax(group_smem<32, 32>(), group_smem<32, 64>()), smax(group_smem<64, 64>(), group_smem<64, 128>())),
         smax(smax(group_smem<128, 128>(), group_smem<128, 256>()), group_smem<256, 256>()));
static_assert(2 * (kGroupSmem + 1024) <= 228 * 1024, "two blocks per SM");

// one tile: the threads past the tile's C L/32 (lengths below 2^13) leave
// before the first barrier, which then waits for the others only
template <int L, int C, bool SEQ_FAST, class Src, class Snk>
__device__ __forceinline__ void group_tile(float2 *smem, const typename Src::Params &sp, const typename Snk::Params &kp,
                                           int tile, int unit) {
    static_assert(C * (L / 32) <= kGroupThreads, "threads of a tile");
    float2 *tw = smem + pass_data_bytes<L, C>() / sizeof(float2);
    fill_twiddles<L>(tw);
    __syncthreads();
    if (threadIdx.x >= C * (L / 32)) return;
    Src src(sp, tile, unit, unit, tw + TwTable<L>::SIZE);
    Snk snk(kp, tile, unit, unit);
    cta_fft<L, C, SEQ_FAST, +1>(smem, tw, src, snk);
    snk.finish(smem);
}

struct GroupPass1 {
    const FilterGroup &p;
    const int s, b;
    float2 *smem;
    template <int N2, int N1>
    __device__ __forceinline__ void run() const {
        constexpr int C = seqs_per_cta<N2>(N1), TILES = N1 / C;
        using Src = TemplateSrc<N2, C, cx_ilog2(N1)>;
        using Snk = ExchSink<N2, C, +1, cx_ilog2(N1)>;
        const GroupSeg &g = p.s[s];
        const typename Src::Params sp{g.seg.W,   p.units + g.unit0, p.anchors + g.anc0, p.anchors4 + g.anc0,
                                      g.max_anc, g.log2D,           0};
        const typename Snk::Params kp{p.exch + g.exch0, g.seg.log2N1, g.seg.log2N};
        group_tile<N2, C, true, Src, Snk>(smem, sp, kp, b % TILES, b / TILES);
    }
};

struct GroupPass2 {
    const FilterGroup &p;
    const int s, b;
    float2 *smem;
    template <int N2, int N1>
    __device__ __forceinline__ void run() const {
        constexpr int C = seqs_per_cta<N1>(N2), TILES = N2 / C;
        using Src = RowSrc<N1, C>;
        using Snk = RhoSink<N1, C>;
        const GroupSeg &g = p.s[s];
        const typename Src::Params sp{p.exch + g.exch0, g.seg.log2N1, g.seg.log2N};
        const typename Snk::Params kp{p.units + g.unit0, p.partials + g.part0, p.staged, p.keys,    p.counter, p.cap,
                                      g.seg.log2N2,      TILES,                g.seg_idx, p.kl};
        group_tile<N1, C, false, Src, Snk>(smem, sp, kp, b % TILES, b / TILES);
    }
};

template <class Op>
__device__ __forceinline__ void group_dispatch(int log2N, const Op &op) {
    switch (log2N) {   // block-uniform
        case 10: op.template run<32, 32>(); break;
        case 11: op.template run<32, 64>(); break;
        case 12: op.template run<64, 64>(); break;
        case 13: op.template run<64, 128>(); break;
        case 14: op.template run<128, 128>(); break;
        case 15: op.template run<128, 256>(); break;
        case 16: op.template run<256, 256>(); break;
    }
}
}  // namespace

// The units and anchors of small banks in one launch: every block of a unit
// forms its UnitInfo anew, by one thread; two launches of 4 and 7 us, 9 us here.
// FP64 bounds it (two operations per SM and clock: 30 a record, and a warp of
// one thread's unit costs as much as one of 32 records), so a block takes 1024
// records where that leaves two blocks per SM: 300 units of 940 records 27.5 us
// in blocks of 256, 22 so.
template <int CAP>
__global__ void __launch_bounds__(kGroupThreads) k_units_anchors(__grid_constant__ const FilterGroupOf<CAP> p) {
    __shared__ UnitInfo su;
    int b = blockIdx.x, i = blockIdx.y;
    chain_wait(b, i);
    if (p.clear && b == 0 && i == 0) clear_ctl(p.clear);
    const int s = CAP > 1 ? group_find(p.end_anc, p.n, b) : 0;
    const GroupSeg &g = p.s[s];
    if (CAP > 1) i = b / g.anc_blocks;
    const int bx = CAP > 1 ? b - i * g.anc_blocks : b;
    const int t = p.order ? p.order[i] : i;
    const double *T = p.tmpl + (int64_t)t * kTmplStride;
    if (threadIdx.x == 0) {
        su = unit_info(g.seg, T, t, p.f_low, p.thr, g.log2D);
        if (bx == 0) p.units[g.unit0 + i] = su;
    }
    __syncthreads();
    const int64_t a0 = g.anc0 + (int64_t)i * g.max_anc;
    unit_anchors(g.seg, T, su, g.log2D, g.max_anc, p.anchors + a0, p.anchors4 + a0, 1, 0, bx, g.anc_blocks);
}

__global__ void __launch_bounds__(kGroupThreads, 2) k_pass1_group(__grid_constant__ const FilterGroup p) {
    extern __shared__ __align__(16) float2 group_shared[];
    int b = blockIdx.x;
    chain_wait(b);
    const int s = group_find(p.end1, p.n, b);
    group_dispatch(p.s[s].seg.log2N, GroupPass1{p, s, b, group_shared});
}

__global__ void __launch_bounds__(kGroupThreads, 2) k_pass2_group(__grid_constant__ const FilterGroup p) {
    extern __shared__ __align__(16) float2 group_shared[];
    int b = blockIdx.x;
    chain_wait(b);
    const int s = group_find(p.end2, p.n, b);
    group_dispatch(p.s[s].seg.log2N, GroupPass2{p, s, b, group_shared});
}

__global__ void __launch_bounds__(kGroupThreads) k_peaks_group(__grid_constant__ const FilterGroup p) {
    int w = (int)((blockIdx.x * kGroupThreads + threadIdx.x) >> 5);
    chain_wait(w);
    if (w >= p.n * p.n_t) return;
    const GroupSeg &g = p.s[w / p.n_t];
    const int i = w % p.n_t, nblk = g.tiles2;
    unit_peak(p.units[g.unit0 + i], p.n_t, p.partials + g.part0 + (int64_t)i * nblk, nblk, g.seg_idx, p.n_seg, p.peaks);
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
// at most eight blocks of 256 threads per SM: beyond, every block's own unit
// costs more than the second launch
bool units_anchors_applies(int n_t, int phase_mode, int n_sm) {
    return phase_mode == MF_PHASE_ANCHOR && n_t <= 8 * n_sm;
}

int group_tiles(int log2N, int n_t, int n_sm) {
    if (log2N < 10 || log2N > 16) return 0;
    const int64_t tiles = (int64_t)n_t << (log2N > 13 ? log2N - 13 : 0);
    return tiles <= 2 * (int64_t)n_sm ? (int)tiles : 0;
}

template <int CAP>
bool group_add(FilterGroupOf<CAP> &p, const SegDev &seg, int seg_idx, int log2D, int max_anc) {
    if (p.n >= CAP) return false;
    GroupSeg &g = p.s[p.n];
    g = GroupSeg{};
    g.seg = seg;
    g.seg_idx = seg_idx;
    g.log2D = log2D;
    g.max_anc = max_anc;
    const int N2 = 1 << seg.log2N2, N1 = 1 << seg.log2N1;
    g.tiles1 = N1 / std::min(8192 / N2, N1);   // columns and rows per tile as in seqs_per_cta
    g.tiles2 = N2 / std::min(8192 / N1, N2);
    g.unit0 = p.n * p.n_t;
    g.anc0 = p.anc_records;
    g.exch0 = p.exch_elems;
    g.part0 = p.n_partials;
    p.anc_records += (int64_t)p.n_t * max_anc;
    p.exch_elems += (int64_t)p.n_t * seg.N;
    p.n_partials += (int64_t)p.n_t * g.tiles2;
    const int at = p.n++;
    p.end1[at] = (at ? p.end1[at - 1] : 0) + p.n_t * g.tiles1;
    p.end2[at] = (at ? p.end2[at - 1] : 0) + p.n_t * g.tiles2;
    return true;
}

template bool group_add(FilterGroupOf<1> &, const SegDev &, int, int, int);
template bool group_add(FilterGroup &, const SegDev &, int, int, int);

template <int CAP>
cudaError_t launch_units_anchors(FilterGroupOf<CAP> &p, int n_sm, cudaStream_t st) {
    if (p.n < 1) return cudaErrorInvalidValue;
    // blocks per unit: of 1024 records, of fewer where that leaves less than two
    // blocks per SM, and at most eight blocks per SM
    const int units = p.n * p.n_t, fill = 2 * n_sm / units, most = std::max(1, 8 * n_sm / units);
    int blocks = 0;
    for (int i = 0; i < p.n; ++i) {
        GroupSeg &g = p.s[i];
        const int fine = (g.max_anc + kGroupThreads - 1) / kGroupThreads, coarse = (fine + 3) / 4;
        g.anc_blocks = std::min(most, std::max(coarse, std::min(fine, fill)));
        p.end_anc[i] = blocks += p.n_t * g.anc_blocks;
    }
    return launch(k_units_anchors<CAP>, CAP > 1 ? dim3(blocks) : dim3(p.s[0].anc_blocks, p.n_t), kGroupThreads, 0, st, p);
}
template cudaError_t launch_units_anchors(FilterGroupOf<1> &, int, cudaStream_t);

cudaError_t launch_group(FilterGroup &p, int n_sm, cudaStream_t st) {
    if (p.n < 1) return cudaErrorInvalidValue;
    for (int i = 0; i < p.n; ++i)
        if (p.s[i].seg.log2N < 10 || p.s[i].seg.log2N > 16 || p.s[i].seg.log2N2 != log2_n2(p.s[i].seg.log2N))
            return cudaErrorInvalidValue;
    cudaError_t e = launch_units_anchors(p, n_sm, st);
    if (e == cudaSuccess) e = launch(k_pass1_group, dim3(p.end1[p.n - 1]), kGroupThreads, kGroupSmem, st, p);
    if (e == cudaSuccess) e = launch(k_pass2_group, dim3(p.end2[p.n - 1]), kGroupThreads, kGroupSmem, st, p);
    const int warps = kGroupThreads / 32;
    if (e == cudaSuccess)
        e = launch(k_peaks_group, dim3((p.n * p.n_t + warps - 1) / warps), kGroupThreads, 0, st, p);
    return e;
}

MF_DEBUG_READER(dbg_read_group)

cudaError_t group_kernel_attributes() {
    cudaError_t e = init_pass_tables();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pass1_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pass2_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupSmem);
    return e;
}

}  // namespace mf
