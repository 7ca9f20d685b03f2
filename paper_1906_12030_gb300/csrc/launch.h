// Kernel launches of the library: each may start while the kernel before it
// on the stream drains (programmatic dependent launch).  Every kernel launched
// so calls pdl_wait() in all its threads before it touches global memory, which
// returns once the kernel before is complete and its writes are visible, and
// pdl_trigger() after that; a kernel that allocates tensor memory does so
// before its trigger, so that no later kernel's blocks can take it first.
// Pointer parameters of these kernels are not __restrict__: that would let
// the compiler read through them before the wait.
// At small bond dimensions a kernel's launch and set-up cost as much as its
// work (chi = 4 ascend: 10 launches, 61 us without the overlap, 44 with it).  `overlap`
// is for kernels whose blocks are all on the GPU at once (each caller's limit
// is what registers and shared memory let it hold); blocks of a larger
// kernel that arrive early take their place from the one before (chi = 12
// OZ4 descend 1.25 -> 1.29 ms).
#pragma once

#include <cuda_runtime.h>

namespace mera {

template <typename... P, typename... A>
void launch(void (*kernel)(P...), bool overlap, dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
            const A&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // its error is the next cudaGetLastError()
}

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Start of a kernel without set-up of its own.
__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  pdl_trigger();
}
#endif

}  // namespace mera
