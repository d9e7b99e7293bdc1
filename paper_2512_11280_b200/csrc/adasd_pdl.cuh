// Programmatic dependent launch, from the kernel's side.
#pragma once

namespace adasd {

// The launch ahead in the stream may still be running when a kernel launched with programmatic
// stream serialisation starts: nothing that launch wrote may be read before pdl_wait().
// pdl_trigger() lets the launch after this one become resident (it waits in its own pdl_wait()).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace adasd
