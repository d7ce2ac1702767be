// Programmatic dependent launch of the solve path's kernels: a kernel launched with
// launch_dep may be scheduled while its predecessor on the stream drains, and waits for the
// predecessor's results in grid_wait(), before it reads or writes memory.  The V-cycle is a chain of
// short dependent kernels; measured on GB300 in a CUDA graph, order-6 float32 half-sweeps in a
// row: 16^3 1.40 -> 1.17 us, 32^3 1.50 -> 1.29, 64^3 2.18 -> 1.93, 128^3 unchanged.  (Letting
// the successor in at the kernel's start instead, so that its waiting blocks take places on
// the SMs, is slower from 32^3 up: 2.15 -> 3.21 us in float64.)
#pragma once

#include <cuda_runtime.h>

namespace mgk {

// Waits until the kernels this one depends on have finished and their writes are visible.
// Every thread of a kernel launched with launch_dep that touches memory calls it before it
// does; what comes earlier (indices, bounds) overlaps the predecessor.
//
// Such a kernel is already running while its inputs are written, so it reads them by plain loads
// through pointers that are not declared __restrict__: the read-only path (__ldg, or const
// __restrict__ parameters) is for data that nobody writes during the kernel's lifetime, and
// neither it nor a restrict pointer has to keep the order with the wait's memory clobber.
// Outputs that a kernel only writes may be __restrict__.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t s, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace mgk
