// Launches that overlap their start with the end of the kernel before them in
// the stream (programmatic dependent launch).  A step of a small lattice takes
// little longer than the gap between two dependent launches: 410 x 200 2.9 -> 2.6 us
// a step, 512^2 4.4 -> 4.1.  No kernel lets the next one start early
// (griddepcontrol.launch_dependents): waiting blocks took slots and issue from
// running ones (410 x 200 3.7 us with it at the start, 2.8 before the stores).
//
// Every kernel launched this way calls chain_wait() before its first access to
// memory that an earlier kernel of the stream writes (or reads: it may be
// written here), so nothing is read early.  Populations, moments and adjoints, which
// the kernels of a chain write, are not read through the non-coherent path: those
// loads could be moved above the wait.  The medium is (__ldg, const __restrict__):
// the calls that write it (lbmp_set_fields, lbmp_batch_set_fields) wait for the stream
// before they return, so no kernel of a chain runs beside its writer.  A path that
// queued a step behind the medium's kernels would have to give that up.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbmp {

// Until the kernels before this one have ended and their writes are visible.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t s, A &&...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}

}  // namespace lbmp
