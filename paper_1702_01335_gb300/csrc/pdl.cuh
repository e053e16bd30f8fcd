// Programmatic dependent launch
#pragma once

namespace lbs {

// Programmatic dependent launch: the stage and finalisation kernels of a stream start while
// their predecessor finishes, do what depends on constants only (descriptor, tables,
// per-velocity values), and wait before they touch anything that a kernel writes.  Every CTA
// waits, also one that then leaves at once, so that a kernel's completion implies that of
// all before it.  A kernel releases its successor late (the stage kernel after its march, the
// finalisation after the cell state): released at the start, the successors of successors
// pile up on the SMs too and a step of the low-Mach runs takes 172 us instead of 115.
static __device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }
static __device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace lbs
