// Programmatic dependent launch of short kernels: the CTAs start while the
// launch before them drains, and wait for it (launch_wait) before they first
// touch global memory, so that back-to-back launches of a few microseconds do
// not pay the launch latency each.  3D FP32 product on 33 x 25 x 29 nodes, one
// after another: 8.2 -> 5.7 us; FP64 energy, gradient, lag and eight products
// on 69 x 45: 100 -> 86 us.  That is the overlap of one launch with the launch
// before it: a single product after other work takes what it did.  Between
// larger kernels the last wave of one and
// the start of the next overlap: the two launches of the 129^3 product 108.6 ->
// 102.9 us, a mixed 129^3 load step (some 3,000 launches) 210 -> 202 ms, the
// five transfers at 129^3 177 -> 168 us, the Galerkin operators of a 65^3
// hierarchy 144 -> 140 us.  The FP64 stencil product, its assembly and the FP64
// gradient and energy passes are launched plainly: on 65 x 49 x 57 energy,
// gradient, lag and eight products took 3,399 us this way against 3,235, and
// nothing was won elsewhere (69 x 45, double-float passes at 97 x 105 x 89).
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace pf {

// Every earlier launch of the stream has ended and its writes are visible
// after this; the launch after this one may then start.  A kernel that calls it
// has no __restrict__ pointers: a load through one could be moved before it,
// also past a branch on a value loaded after it.
__device__ __forceinline__ void launch_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The same, and the block's index as a value that is known only after the wait:
// an address worked out from it cannot be read earlier, __restrict__ or not.
__device__ __forceinline__ unsigned launch_wait_block() {
  unsigned zero = 0;
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" : "+r"(zero)::"memory");
  return blockIdx.x + zero;
}

// Launch of a kernel whose threads call launch_wait() before any global memory
// access.  An ordinary launch under stream capture (the CG graphs' bodies).
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                    A&&... a) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
    cudaGetLastError();
    cap = cudaStreamCaptureStatusActive;
  }
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, std::forward<A>(a)...);
}

template <class... P, class... A>
inline cudaError_t launch_dependent(void (*k)(P...), dim3 grid, dim3 block, cudaStream_t st, A&&... a) {
  return launch_dependent(k, grid, block, size_t(0), st, std::forward<A>(a)...);
}

}  // namespace pf
