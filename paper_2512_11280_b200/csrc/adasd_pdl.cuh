// Programmatic dependent launch, from the kernel's side.
#pragma once

namespace adasd {

// The launch ahead in the stream may still be running when a kernel launched with programmatic
// stream serialisation starts: nothing that launch wrote may be read before pdl_wait().
// Nor may it be read through the non-coherent path, which wants data that nobody writes while this launch is
// resident: whatever the caller or another call passes in (logits, windows, tokens, uniforms, cutoffs) may have been
// written by the launch ahead.  Kernels use plain loads or __ldcg.
// pdl_trigger() lets the launch after this one become resident (it waits in its own pdl_wait()).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace adasd
