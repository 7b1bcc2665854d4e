// Programmatic dependent launch for chains of short kernels (a line search, the inverses and the products of
// the refreshes): a kernel's launch and prologue (barriers, tensor memory) lie beside the last CTAs of the kernel
// before it instead of after it. Every kernel launched
// this way calls dev::pdl_begin() before it touches memory that earlier kernels write or read: it waits until
// they are complete and their writes are visible. No kernel lets the next one start before its CTAs exit: an
// early start fills SMs that happen to have room, and the float64-bound products then ran up to 15 % slower. A
// line search is a chain of eleven kernels; by this alone a float64 solve of m = 207, n = 36 with gradients went from
// 8.8 to 7.0 ms, of m = 416, n = 64 from 9.0 to 7.8. The inverses are longer chains: float64-class inverse of
// m = 3328 15.2 -> 13.9 ms, mixed solve of m = 1495, n = 260 (float64 inverse) 20.8 -> 20.2.
#pragma once
#include <cuda_runtime.h>

#include <utility>

#include "omm_internal.cuh"

namespace omm {
namespace dev {
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
}  // namespace dev

template <typename... P, typename... A>
void launch_pdl(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(P...), A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  OMM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...));
}

}  // namespace omm
