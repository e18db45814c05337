// pdl.cuh -- kernels of one stream launched as programmatic dependents: the
// next kernel's blocks are scheduled while this one's last blocks still run,
// which hides the gap between two grids (about a microsecond, against the 3-20
// us of most of the network's kernels).  Training step of 16 fields of 256 x 64
// 952 -> 901 us, of 8 fields of 512 x 128 1400 -> 1341 us, warm start of a 2048 x
// 512 lattice 899 -> 844 us; initial state, 100 steps and moments of a 512 x 256
// lattice 994 -> 975 us.
//
// begin() is the first statement of every kernel that launch() starts (the sweep
// kernels have a wait of their own, after their set-up).  It waits
// until the grid before has finished and its writes are visible, and only then
// lets the next grid be scheduled; so whatever came earlier on the stream is
// complete when any block passes it, and a block that waits holds no tensor
// memory.
#pragma once

#include <cuda_runtime.h>

namespace pdl {

__device__ __forceinline__ void begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace pdl
