// Device side of programmatic dependent launch.
#pragma once

namespace fcgle {

// Every kernel launched with launch_pdl (tma_host.h) lets the next kernel of its
// stream be scheduled as soon as all of its own CTAs are running (pdl_trigger at
// entry) and, after its prologue, waits until the previous kernel of the stream
// has completed and its writes are visible (pdl_wait) before it touches global
// memory that another kernel writes.  The wait ends when that kernel ends;
// without the launch attribute both are no-ops.
//
// Such a kernel is alive while its predecessors still write, so it must not read
// their results through the read-only path (ld.global.nc, which is defined only
// for data that nothing writes during the kernel): neither __ldg nor const
// __restrict__ parameters, from which the compiler may make the same loads.
// Constants of the handle, complete before setup returns, may be read so.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter() {
  pdl_trigger();
  pdl_wait();
}

}  // namespace fcgle
