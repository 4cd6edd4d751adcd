// Launches that overlap a kernel's launch and set-up with the end of the kernel before it on the stream
// (programmatic dependent launch), and the device-side half every kernel of the library executes.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace sl {

// Executed by every thread of every kernel launched with launch_overlapped, after set-up that touches no global
// memory and before anything that does: waits until the kernel before this one on the stream has completed and its
// writes are visible, then lets the next kernel's blocks be placed as this one's leave room.  The order matters
// twice: the next kernel starts only after this one's wait, so everything older is complete by then; and a kernel
// that allocates tensor memory does so before this call, so that a block of the next kernel can never hold columns
// that a block of this one still waits for.  Without the launch attribute both instructions do nothing.
__device__ __forceinline__ void overlap_sync() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Whether the operation before the next launch of this thread is a kernel that this same call of the library put on
// the same stream.  Only then may a launch overlap it: griddepcontrol.wait is defined by the grids before a kernel,
// not by copies, memsets or other work of the caller.  Every entry point that launches starts a chain of its own, and
// a copy or memset between two kernels breaks it.
extern thread_local bool t_in_chain;
extern thread_local int64_t t_launches;      // kernels launched by this thread
inline void break_chain() { t_in_chain = false; }
struct LaunchChain {
  LaunchChain() { t_in_chain = false; }
  ~LaunchChain() { t_in_chain = false; }
};
// Attributes of the next launch, `at` with room for one more after `n`; returns their number.
inline unsigned chain_attribute(cudaLaunchAttribute* at, unsigned n) {
  ++t_launches;
  if (!t_in_chain) { t_in_chain = true; return n; }
  at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[n].val.programmaticStreamSerializationAllowed = 1;
  return n + 1;
}

// kernel<<<grid, block, smem, st>>>(args...), starting early where the chain allows.  Most of a round over few
// tokens is launches of 3-6 us each, of which the gap to the kernel before and the set-up were 1.5-2 us: a
// GPT-2-medium-shaped round of 512 tokens 4.88 -> 3.81 ms (586 launches then).
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  cfg.attrs = at; cfg.numAttrs = chain_attribute(at, 0);
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace sl
