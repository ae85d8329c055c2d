// launch.cuh -- launches that overlap a kernel's start with the end of the kernel before it in the stream.
//
// A build is a chain of short dependent kernels (18 launches of 4 to 15 us for a 256^2 cell).  Launched
// with programmatic stream serialisation, the CTAs of the next kernel take the SMs as the last CTAs of
// this one leave and run their prologue (twiddles into shared memory, barriers, tables), then wait in
// after_previous() until the kernel before has finished and its stores are visible.  Every kernel of such
// a chain calls both: next_may_start() at its top, after_previous() before it touches anything that another
// kernel writes or that the kernel before may still read.  (A kernel may start before the kernels ahead of
// its predecessor have finished: what a prologue reads must have been complete before the chain began, at a
// plain launch or a copy.)
// Measured: S-matrix build of a 256^2 cell 195 -> 152 us, multislice of 256 probes there 676 -> 624 us, a
// 512^2 simulation (120 us passes of 56 M points) 3.92 -> 3.84 ms; no difference at 1024^2 with 129 beams
// (200 to 300 us passes of 135 M points), and 15.28 -> 15.50 ms for an 8-slice build of 529 beams there (0.8
// and 1.2 ms passes).  So the passes chain up to CHAIN_POINTS points.
// Under stream capture the launches are plain ones.
#pragma once
#include <cuda_runtime.h>

namespace prism {

__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

constexpr long long CHAIN_POINTS = 1LL << 26;

template <class... P, class... A>
static cudaError_t launch_chained_if(bool chain, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (chain && cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();  // (as if captured: a plain launch)
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, args...);
}
template <class... P, class... A>
static cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args) {
    return launch_chained_if(true, kernel, grid, block, smem, s, args...);
}

}  // namespace prism
