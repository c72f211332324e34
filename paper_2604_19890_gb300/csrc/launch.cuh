// Launches that overlap the start of a kernel with the end of the one before it
// on the stream (programmatic dependent launch). A kernel launched with
// launch_early may have its blocks resident while its predecessor's last blocks
// still run, so it begins with enter_grid(), before any return and before any
// access to memory that an earlier kernel writes or reads: it lets the next
// kernel start early in turn and then waits until every earlier grid of the
// stream has completed and its writes are visible (each grid waits for its
// predecessor, so the order is the stream's order throughout). Kernels without
// enter_grid are launched the plain way and wait for complete predecessors.
// The key switch of a small ring is a chain of a dozen kernels of a few
// microseconds each, whose launch gaps this hides: by itself it takes a query at
// N = 2^13 from 4.50 ms to 4.19, a rotate-sum at N = 2^15 from 652 us to 611 and one
// multiplication at N = 2^13 from 69.6 us to 68.6. Blocks that wait early hold
// room that kernels of other streams could use, so a thread that feeds one of
// several streams side by side launches the plain way (PlainLaunches): the mixed
// batch on three streams took 11.1 ms with early launches and 10.8 without.
#pragma once
#include <cuda_runtime.h>

#include <utility>

#include "ss_internal.h"

namespace ss {

__device__ __forceinline__ void enter_grid() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
void launch_early(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = plain_launches() ? 0 : 1;
  SS_CUDA(cudaLaunchKernelEx(&c, kernel, static_cast<P>(std::forward<A>(args))...));
}

}  // namespace ss
