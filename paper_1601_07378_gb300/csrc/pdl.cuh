// pdl.cuh -- programmatic dependent launch of the chain's kernels.
//
// The passes of an apply are short dependent launches on one stream (5 to 10 us
// each for a few bands), so the launch latency between them counts.  A kernel
// launched by pdl_launch() may be set up while its predecessor in the stream
// drains; it must start with pdl_begin(), which waits until everything before
// it has completed and is visible, before it touches memory.  (A kernel that
// begins so may also be launched the ordinary way.)  It is resident while its
// predecessors still write, so what the caller passes or an earlier launch
// leaves (coefficients, V, diag, occupations, cylinder, dense rows, partial
// sums) is not read-only for its lifetime: its parameters for them are not
// `const __restrict__`, which would let the compiler read them by the
// non-coherent path or above the wait, and its inline loads of them are
// volatile with a memory clobber.  Tables and twiddles, complete when the plan
// is made, may be.  Neither costs anything: twelve workloads from 24^3 x 1 to
// 96^3 x 1024 bands took the same time to 0.1 % with and without.
// No kernel triggers its successor early: blocks that wait take their place on
// the SMs unevenly while the predecessor runs, which measured slower everywhere.
// us per apply, calls back to back, without the attribute / with it (with an
// early trigger where the same chain was timed):
//   FP32  five launches  24^3 x 1  22.6 / 12.4    48^3 x 8   26.0 / 15.3
//         the line path  24^3 x 40 18.5 / 10.1    48^3 x 20  22.9 / 16.0 (20.6)
//                        96^3 x 8  43.1 / 35.2 (41.6)   96^3 x 512 1618 / 1609 (1726)
//   FP64  24^3 x 1  34.9 / 24.7 (25.4)    48^3 x 4   79.7 / 68.0 (87 to 156)
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace vloc {

__device__ __forceinline__ void pdl_begin() { cudaGridDependencySynchronize(); }

template <class... P, class... A>
inline int pdl_launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here, not by a later check
    return (int)e;
}

}  // namespace vloc
