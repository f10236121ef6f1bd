// mf_launch.h -- launches chained within a call (programmatic dependent launch).
//
// A call on a short segment is a chain of kernels of 3 .. 10 us with 1.5 us and
// more between the end of one and the first instruction of the next.  Inside a
// ChainScope the launches carry the programmatic-serialization attribute, and
// every kernel launched with it waits for its predecessor itself (chain_wait),
// so its launch, its twiddle copies and its barrier set-up run under the end of
// the one before: a 16-template search step on 2^16 samples 63 -> 45 us, four
// short segments 228 -> 163.  No kernel triggers its successor early
// (griddepcontrol.launch_dependents): CTAs waiting from the start hold places
// that the predecessor's successors need (79, 208 us).
//
// Rules.  Every kernel passed to launch() executes chain_wait in all threads,
// before the first access to anything another kernel of a call writes or reads
// (constant tables of the library may be read before it): a kernel then
// completes only after its predecessor has, so the order along the chain is
// that of plain launches.  chain_wait takes the indices (or pointers) that
// every later global address depends on and hands them back opaque: a read-only
// load (__ldg, or through a const __restrict__ parameter) of what the
// predecessor writes may otherwise be moved above the wait, since the compiler
// takes such memory to be constant.  Without the attribute chain_wait is a
// no-op.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace mf {

inline thread_local bool t_chain = false;   // set for the duration of a call by ChainScope
struct ChainScope {
    const bool before;
    explicit ChainScope(bool on) : before(t_chain) { t_chain = on; }
    ~ChainScope() { t_chain = before; }
    ChainScope(const ChainScope &) = delete;
    ChainScope &operator=(const ChainScope &) = delete;
};

// in clusters of `cluster` CTAs along x (0: none)
template <class... P, class... A>
inline cudaError_t launch_in_clusters(void (*kernel)(P...), dim3 grid, unsigned threads, unsigned cluster, size_t smem,
                                  cudaStream_t st, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    cfg.attrs = at;
    if (t_chain) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[cfg.numAttrs].val.clusterDim.x = cluster;
        at[cfg.numAttrs].val.clusterDim.y = 1;
        at[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A &&...args) {
    return launch_in_clusters(kernel, grid, threads, 0, smem, st, std::forward<A>(args)...);
}

__device__ __forceinline__ void chain_opaque(int &x) { asm volatile("" : "+r"(x)::"memory"); }
__device__ __forceinline__ void chain_opaque(int64_t &x) { asm volatile("" : "+l"(x)::"memory"); }
template <class T>
__device__ __forceinline__ void chain_opaque(T *&x) {
    asm volatile("" : "+l"(x)::"memory");
}
template <class... I>
__device__ __forceinline__ void chain_wait(I &...index) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (chain_opaque(index), ...);
}
// before the first asynchronous copy of memory the predecessor wrote
template <class... I>
__device__ __forceinline__ void chain_wait_async(I &...index) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("fence.proxy.async;" ::: "memory");
    (chain_opaque(index), ...);
}

}  // namespace mf
