// rlb_launch.cuh -- launching a kernel while the grid before it in its stream drains.
#pragma once
#include <cuda_runtime.h>

namespace {

// A step kernel is launched while the grid before it in the stream drains (launch_after):
// this waits until that grid is complete and its writes are visible.  The pointers pass
// through, so that no load from them can be moved up (a memory clobber alone does not hold
// back loads from __restrict__ pointers): every pointer that a kernel reads through goes
// here.  They are read with coherent loads, since the grid before writes while this kernel
// is already resident.
template <typename T>
__device__ __forceinline__ void wait_for_grid(const T* __restrict__& p) {
  asm volatile("griddepcontrol.wait;" : "+l"(p)::"memory");
}
template <typename T>
__device__ __forceinline__ void wait_for_grid(T* __restrict__& p) {
  asm volatile("griddepcontrol.wait;" : "+l"(p)::"memory");
}
template <typename T>
__device__ __forceinline__ void wait_for_grid(const T* __restrict__& p, const T* __restrict__& q) {
  asm volatile("griddepcontrol.wait;" : "+l"(p), "+l"(q)::"memory");
}

// Launch of a step kernel while the grid before it in the stream drains: the kernel waits for
// that grid itself (wait_for_grid), so that only its launch latency overlaps, 2-3 us of every
// step: 16 x 20 x 24 FP64 8.3 -> 5.3 us per step, 32^3 16.4 -> 13.4, FP32 storage 6.3 -> 3.8,
// 64^3 FP32 16.5 -> 14.9, 256^3 FP64 1798.8 -> 1796.5, D2Q9 4 x 800 with C_7 12.4 -> 9.3.
// early = false: an ordinary launch (a stream that has just waited for another one).
template <typename... P, typename... A>
void launch_after(dim3 grid, int block, cudaStream_t st, bool early, void (*kernel)(P...), A... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.blockDim = dim3((unsigned)block);
  lc.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  lc.attrs = &at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, kernel, P(args)...);
}

}  // namespace
