// Programmatic dependent launch along a call's kernels: a kernel launched with it is scheduled while its
// predecessor runs and does what needs no data (barriers, tensor memory) before pdl_wait(), which returns
// once every earlier kernel of the stream has completed.  Every kernel that may be launched so calls
// pdl_wait() in all its threads' paths before anything else touches global memory, and before any return
// (a kernel whose blocks all left without waiting would let its successor run ahead of its predecessor).
//
// Small frames only (kPdlAtoms): there a step is a chain of kernels that each leave most SMs idle, and the
// chain of launches is a good part of it.  On large frames the waiting blocks of the next kernel hold
// shared memory and registers of SMs that the running one still needs.  Steps without and with it, FP32: 540 atoms 270
// and 242 us, 1,029 298 and 285, 3,267 339 and 304, 4,356 365 and 333, 8,232 471 and 446, 12,288 508 and 513; mixed
// mode: 1,029 228 and 215, 3,267 262 and 268, 8,232 319 and 316, 12,288 386 and 376.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace dpgb {

constexpr long kPdlAtoms = 4096;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... KA, class... A>
cudaError_t launch_chain(bool pdl, void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace dpgb
