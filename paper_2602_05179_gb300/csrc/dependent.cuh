// dependent.cuh -- programmatic dependent launch within one operator call.
//
// The kernels of a call run one after the other on the caller's stream, and a
// small call is mostly the time between them: each launch waits for the whole
// grid before it, then places its blocks, then sets up shared memory.  A kernel
// launched with launch_dependent is placed while its predecessor still runs
// and stops at dep_wait() until that one has completed with all its writes
// visible (n = 50, S = 1,000: 28.8 -> 23.6 us of device time; n = 333, 50,001
// scenarios with predecessors: 135 -> 130).  The recomputation of flagged
// scenarios is launched the ordinary way: placed early, its one busy warp ran
// slower (soft capacity, n = 500, S = 200,000: 454 -> 483 us).
//
// Rules that make this safe:
//  - every thread of such a kernel calls dep_wait() before it touches global
//    memory, so the grid cannot complete before its predecessor has, and what
//    holds for the predecessor's predecessor follows;
//  - the first kernel of a call is launched the ordinary way: nothing of a call
//    starts before all earlier work of the stream is done;
//  - memory that an earlier kernel of the call writes is not read through
//    __restrict__ pointers or __ldg at an address known before dep_wait():
//    such loads may be moved across it.
// dep_launch() lets the next kernel be placed once every block has called it
// (or has ended); a kernel without it does so by ending.
#pragma once

#include "sdp_internal.cuh"

namespace sdp {

__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// dependent = false: an ordinary launch (dep_wait() then does nothing), where
// the stream's previous operation is a copy or a timing event
template <typename... P, typename... A>
cudaError_t launch_dependent(bool dependent, void (*k)(P...), int grid, int block, size_t smem, cudaStream_t st,
                             A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = dependent ? 1u : 0u;
  return cudaLaunchKernelEx(&c, k, P(args)...);
}

}  // namespace sdp
