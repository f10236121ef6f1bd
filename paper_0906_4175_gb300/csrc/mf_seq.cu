// mf_seq.cu -- batched complex FFT of sequences of 4096, 8192 and 16384 points,
// one kernel per call: a sequence stays in one CTA's shared memory through
// three Stockham stages (radix 32, 32 and N/1024), so every point is read and
// written once.  Through the four-step passes these lengths moved twice the
// bytes and the second pass stored through a bank-conflicted tile: 1000
// transforms of 16384 points took 129 us, 71 us here (3.7 TB/s, 0.55 of the
// copy bandwidth; one CTA of 16 warps per SM cannot hide all of its barriers).
//
// Bound: HBM (16 bytes a point).  A CTA works through the batch with a stride;
// as soon as its last stage has read shared memory, every thread starts the
// asynchronous copies of exactly those points of the next sequence that it
// will itself load in stage 0, so they land under the last stage's arithmetic
// and stores and no barrier is needed for them.  256 threads and two CTAs per
// SM for 4096 (two sequences each) and 8192 points, one CTA of 512 threads for
// 16384 (132 KB of data).
//
// Twiddles: stage 1 from a 32 x 32 table in shared memory; stage 2 keeps the
// rows r = 1, 2, 4, 8 of exp(2 pi i r k / N), k < 1024, and forms the others as
// products of at most four of them (all 15 rows of 16384 points would be 120 KB).
#include <algorithm>

#include "mf_fft.cuh"
#include "mf_internal.h"

namespace mf {
namespace {

template <int L>
struct SeqShape {
    static constexpr int T = L / 32;              // threads per sequence
    static constexpr int C = L == 4096 ? 2 : 1;   // sequences per CTA
    static constexpr int R2 = L / 1024;           // radix of the last stage
    static constexpr int ROWS = cx_ilog2(R2);     // twiddle rows r = 1, 2, 4, ..
    static constexpr int STRIDE = L + L / 32;
    static constexpr int NT = C * T;
    static constexpr int PER_SM = NT <= 256 ? 2 : 1;
    static constexpr size_t SMEM = ((size_t)C * STRIDE + 1024 + ROWS * 1024) * sizeof(float2);
};
// rows of 4096 points, then 8192, then 16384
template <int L>
__host__ __device__ constexpr int seq_tw_offset() {
    if constexpr (L == 4096) return 0;
    else return seq_tw_offset<L / 2>() + SeqShape<L / 2>::ROWS * 1024;
}
constexpr int kSeqTwTotal = seq_tw_offset<16384>() + SeqShape<16384>::ROWS * 1024;
static __device__ float2 g_seq_tw1[1024];             // exp(2 pi i r k / 1024) at r * 32 + k
static __device__ float2 g_seq_tw2[kSeqTwTotal];      // exp(2 pi i 2^h k / L) at h * 1024 + k

template <int L>
__device__ void seq_fill_rows() {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < SeqShape<L>::ROWS * 1024; m += gridDim.x * blockDim.x)
        g_seq_tw2[seq_tw_offset<L>() + m] = unit_root<+1>((uint32_t)(m & 1023) << (m >> 10), cx_ilog2(L));
}
__global__ void k_init_seq_tw() {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < 1024; m += gridDim.x * blockDim.x)
        g_seq_tw1[m] = unit_root<+1>((uint32_t)((m >> 5) * (m & 31)), 10);
    seq_fill_rows<4096>();
    seq_fill_rows<8192>();
    seq_fill_rows<16384>();
}

__device__ __forceinline__ void seq_copy8(float2 *dst, const float2 *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int L, int SIGN>
__global__ void __launch_bounds__(SeqShape<L>::NT, SeqShape<L>::PER_SM)
    k_fft_seq(const float2 *x, float2 *y, int64_t n_seq) {
    using S = SeqShape<L>;
    constexpr int T = S::T, R2 = S::R2, NB = 32 / R2;
    extern __shared__ float2 seq_smem[];
    float2 *tw1 = seq_smem + S::C * S::STRIDE, *tw2 = tw1 + 1024;
    for (int m = threadIdx.x; m < 1024; m += S::NT) tw1[m] = __ldg(&g_seq_tw1[m]);
    for (int m = threadIdx.x; m < S::ROWS * 1024; m += S::NT) tw2[m] = __ldg(&g_seq_tw2[seq_tw_offset<L>() + m]);
    const int q = threadIdx.x / T, t = threadIdx.x % T;
    float2 *sq = seq_smem + q * S::STRIDE;
    auto start = [&](int64_t s) {   // this thread's points of sequence s (if there is one)
        if (s < n_seq) {
            const float2 *src = x + s * L + t;
#pragma unroll
            for (int r = 0; r < 32; ++r) seq_copy8(&sq[t + r * T], src + r * T);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int64_t step = (int64_t)gridDim.x * S::C;
    start((int64_t)blockIdx.x * S::C + q);
    for (int64_t s0 = (int64_t)blockIdx.x * S::C; s0 < n_seq; s0 += step) {
        const int64_t s = s0 + q;
        const bool act = s < n_seq;
        float2 v[32];
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // a slot without a sequence runs on zeros
#pragma unroll
        for (int r = 0; r < 32; ++r) v[r] = act ? sq[t + r * T] : czero();
        Dft<32, SIGN>::run(v);
        __syncthreads();   // every thread has its points (first round: the tables are there too)
#pragma unroll
        for (int r = 0; r < 32; ++r) sq[spad(32 * t + r)] = v[r];
        __syncthreads();
        {   // stage 1: radix 32 over Ns = 32
            const int k = t & 31;
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = sq[spad(t + r * T)];
#pragma unroll
            for (int r = 1; r < 32; ++r) {
                float2 w = tw1[r * 32 + k];
                if (SIGN < 0) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
            Dft<32, SIGN>::run(v);
            __syncthreads();
            const int d = (t >> 5) * 1024 + k;
#pragma unroll
            for (int r = 0; r < 32; ++r) sq[spad(d + r * 32)] = v[r];
        }
        __syncthreads();
        // stage 2: radix R2 over Ns = 1024, butterflies b = t + i T
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
            for (int r = 0; r < R2; ++r) v[i * R2 + r] = sq[spad(t + i * T + r * 1024)];
        __syncthreads();   // shared memory is free
        start(s + step);
        float2 *out = y + s * L + t;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            float2 w[R2];
#pragma unroll
            for (int r = 1; r < R2; ++r) {
                if ((r & (r - 1)) == 0) {
                    w[r] = tw2[cx_ilog2(r) * 1024 + t + i * T];
                    if (SIGN < 0) w[r].y = -w[r].y;
                } else {
                    const int top = 1 << cx_ilog2(r);
                    w[r] = cmul(w[top], w[r - top]);
                }
                v[i * R2 + r] = cmul(v[i * R2 + r], w[r]);
            }
            Dft<R2, SIGN>::run(v + i * R2);
            if (act) {
#pragma unroll
                for (int r = 0; r < R2; ++r) __stcs(&out[i * T + r * 1024], v[i * R2 + r]);
            }
        }
    }
}

int g_seq_sms = 0;

template <int L, int SIGN>
cudaError_t seq_run(const float2 *x, float2 *y, int64_t n, cudaStream_t st) {
    using S = SeqShape<L>;
    const int64_t need = (n + S::C - 1) / S::C;
    const unsigned grid = (unsigned)std::min<int64_t>(need, (int64_t)S::PER_SM * g_seq_sms);
    k_fft_seq<L, SIGN><<<grid, S::NT, S::SMEM, st>>>(x, y, n);
    return cudaGetLastError();
}
template <int L>
cudaError_t seq_attrs() {
    cudaError_t e = cudaFuncSetAttribute(k_fft_seq<L, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)SeqShape<L>::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_fft_seq<L, +1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SeqShape<L>::SMEM);
}

}  // namespace

bool fft_seq_applies(int64_t N) { return N == 4096 || N == 8192 || N == 16384; }

cudaError_t launch_fft_seq(const float2 *x, float2 *y, int64_t N, int64_t batch, int sign, cudaStream_t st) {
    switch (N) {
        case 4096: return sign < 0 ? seq_run<4096, -1>(x, y, batch, st) : seq_run<4096, +1>(x, y, batch, st);
        case 8192: return sign < 0 ? seq_run<8192, -1>(x, y, batch, st) : seq_run<8192, +1>(x, y, batch, st);
        case 16384: return sign < 0 ? seq_run<16384, -1>(x, y, batch, st) : seq_run<16384, +1>(x, y, batch, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t seq_kernel_attributes() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_seq_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = seq_attrs<4096>();
    if (e == cudaSuccess) e = seq_attrs<8192>();
    if (e == cudaSuccess) e = seq_attrs<16384>();
    if (e != cudaSuccess) return e;
    k_init_seq_tw<<<8, 256>>>();
    e = cudaGetLastError();
    return e == cudaSuccess ? cudaDeviceSynchronize() : e;
}

}  // namespace mf
